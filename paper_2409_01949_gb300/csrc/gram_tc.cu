// Gram blocks G_ij = M_i^T M_j on the tcgen05 tensor cores (BF16 in, FP32
// accumulation in TMEM).
//
// The Gram matrix of the least-squares system (normal equations of Eq.
// multilevel_ls) inherits the block structure of Eq. multilevel_domain_decomp:
// G_ij is nonzero only when the supports of subdomains i and j share
// collocation points, and then it is a dense K x K contraction over those
// rows.  With rows sorted by cells, the shared rows of a pair are a list of
// runs (one per shared cell, merged where both panels continue contiguously),
// each a multiple of 16 rows.
//
// Operands come from the BF16 copy of the panels written by the assembly kernel in
// mixed precision, laid out as the tensor cores read it: per 16 panel rows one
// block of 8 x 8 core matrices (8 features x 8 rows, 128 contiguous bytes),
// features fastest, then the two row halves.  For one pair, A = P_i^T (features x
// rows) and B = P_j^T are both K-major along the contraction; a box of up to 128
// rows (256 at K <= 32) is one contiguous bulk copy into a shared-memory ring, and each of its 16-row
// blocks one MMA step without swizzle.  One thread issues tcgen05.mma (M = 128,
// N = K rounded up to 16) into a TMEM accumulator, releasing each stage with
// tcgen05.commit.  Feature rows of a tile past K hold whatever the ring holds:
// they reach only accumulator rows and columns past K, which are never read.
// (As a feature-major matrix, 64-row boxes of it read by 2-D TMA were 128-byte
// pieces 4 MB apart: 4.3 GB of DRAM reads for 0.57 GB of panels at 400^2 points,
// K = 128, at a third of the DRAM rate.)
//
// One persistent CTA per SM walks its list of pairs: a producer warp, an MMA warp
// and four epilogue warps, with two accumulators, so that the ring runs on across
// pairs while the last one's block is stored.  A pair is one accumulation chain over
// its rows in cell order, so that its block depends on its own rows only: the tensor
// cores truncate each step's sum, and a chain cut by the system's size would move a
// block by up to 5e-5 of its norm from system to system.  The longest chain (level 1
// with itself: 1263 boxes of one CTA) takes about as long as all CTAs' shares.
// Large pairs are dealt first, the rest in the order of their first cell, each to
// the CTA with the least work so far, so that all CTAs are in the same place at the
// same time and the panels stay in L2.  400^2 points, levels 1..16, K = 128 (6297
// pairs), against one CTA per pair, pair after pair: 1.64 -> 0.79 ms, 330 -> 690
// TFLOP/s; 2048^2, levels 1..64, K = 64: 49.6 -> 33.8 ms, 170 -> 249 TFLOP/s (half of
// each MMA's rows are past K there).
//
// Every mbarrier wait is bounded; a timeout raises flags[2].
#include <algorithm>
#include <cstring>
#include <functional>
#include <queue>

#include <new>
#include <stdexcept>

#include "elmfb_internal.cuh"
#include "sm100_ptx.cuh"

namespace {

constexpr int kMaxGramStages = 12;
constexpr int kGramThreads = 192;            // producer, MMA, four epilogue warps
constexpr size_t kGramRing = 192 * 1024;
// ring, 1 KB alignment, and the rest of a 128-row tile past the last stage's K rows
constexpr size_t kGramSmem = kGramRing + 16 * 1024 + 1024;

// Contraction rows per box.  A box costs the producer and the MMA thread about 700
// cycles whatever its size (boxes of 64 rows took the same time at K = 64 and K =
// 128, and half the ring cost 4%), so it is as large as leaves three stages or more
// of the ring: 64 -> 128 rows took 0.94 -> 0.75 ms at K = 128, 45.6 -> 33.4 ms at K =
// 64 on the workloads above (with their pairs cut).
__host__ __device__ constexpr int gram_box_rows(int K) { return K <= 32 ? 256 : 128; }
__host__ __device__ constexpr int gram_tile_bytes(int K) {
  return gram_box_rows(K) / 16 * gram_block_bytes(K);
}

// device memory that blocks on their way to the host pass through
constexpr int64_t kGramStaging = 32 << 20;

// tasks: (first run, end run, 2 boxes + diagonal, block of G)
__global__ void __launch_bounds__(kGramThreads, 1)
    k_gram_tc(const uint8_t* __restrict__ pt, const int4* __restrict__ tasks,
              const int* __restrict__ task_off, const int4* __restrict__ runs, int K, int N, int S,
              float* __restrict__ G, int* __restrict__ flags) {
  extern __shared__ uint8_t smraw[];
  __shared__ __align__(8) uint64_t full[kMaxGramStages];
  __shared__ __align__(8) uint64_t empty[kMaxGramStages];
  __shared__ __align__(8) uint64_t acc_full[2], acc_empty[2], done;
  __shared__ uint32_t tmem_slot;
  uint8_t* sm = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smraw) + 1023) & ~uintptr_t(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int box = gram_box_rows(K);
  const int tile_bytes = gram_tile_bytes(K), block_bytes = gram_block_bytes(K);
  const int t0 = task_off[blockIdx.x], t1 = task_off[blockIdx.x + 1];   // this CTA's tasks

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      sm100::mbar_init(&full[s], 1);
      sm100::mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      sm100::mbar_init(&acc_full[b], 1);
      sm100::mbar_init(&acc_empty[b], 4);   // one arrival per epilogue warp
    }
    sm100::mbar_init(&done, 1);
    sm100::fence_mbar_init();
  }
  if (warp == 2) sm100::tmem_alloc(&tmem_slot, 256);
  sm100::tc_fence_before();
  __syncthreads();
  sm100::tc_fence_after();
  const uint32_t tmem = tmem_slot;
  bool ok = true;

  if (warp == 0 && lane == 0) {
    // producer: box b goes to stage b mod S once box b - S has left it
    int st = 0, ph = 1, issued = 0;
    for (int t = t0; t < t1 && ok; ++t) {
      const int4 task = tasks[t];
      const bool diag = task.z & 1;
      int4 next = runs[task.x];   // one record ahead, so that its load is not waited for
      for (int r = task.x; r < task.y && ok; ++r) {
        const int4 run = next;
        next = runs[min(r + 1, task.y - 1)];
        for (int off = 0; off < run.z; off += box) {
          if (!sm100::mbar_wait(&empty[st], ph)) {   // the first round passes at once
            ok = false;
            break;
          }
          uint8_t* a = sm + (size_t)st * 2 * tile_bytes;
          const uint32_t bytes = (uint32_t)(min(box, run.z - off) / 16 * block_bytes);
          sm100::mbar_arrive_expect_tx(&full[st], diag ? bytes : 2 * bytes);
          sm100::bulk_load(a, pt + (int64_t)((run.x + off) >> 4) * block_bytes, bytes, &full[st]);
          if (!diag)
            sm100::bulk_load(a + tile_bytes, pt + (int64_t)((run.y + off) >> 4) * block_bytes,
                             bytes, &full[st]);
          ++issued;
          if (++st == S) {
            st = 0;
            ph ^= 1;
          }
        }
      }
    }
    // no copy of this CTA is left in flight when it ends
    for (int b = max(0, issued - S); b < issued; ++b)
      if (!sm100::mbar_wait(&full[b % S], (b / S) & 1)) ok = false;
    if (!ok) atomicOr(&flags[2], 1);
  } else if (warp == 1 && lane == 0) {
    // MMA issuer: task q of this CTA accumulates in TMEM buffer q mod 2
    const uint32_t idesc = sm100::idesc_bf16_f32(128, N);
    int st = 0, ph = 0, q = 0;
    for (int t = t0; t < t1 && ok; ++t, ++q) {
      const int4 task = tasks[t];
      const int buf = q & 1;
      if (!sm100::mbar_wait(&acc_empty[buf], ((q >> 1) & 1) ^ 1)) {
        ok = false;
        break;
      }
      sm100::tc_fence_after();
      const uint32_t acc_at = tmem + (uint32_t)buf * 128u;
      uint32_t acc = 0;
      int next = runs[task.x].z;
      for (int r = task.x; r < task.y && ok; ++r) {
        const int len = next;
        next = runs[min(r + 1, task.y - 1)].z;
        for (int off = 0; off < len; off += box) {
          if (!sm100::mbar_wait(&full[st], ph)) {
            ok = false;
            break;
          }
          sm100::tc_fence_after();
          const uint8_t* a = sm + (size_t)st * 2 * tile_bytes;
          const uint32_t lead = (uint32_t)block_bytes / 2;   // between the row halves
          const uint64_t ad = sm100::sdesc_k_plain(sm100::smem_u32(a), lead, 128);
          const uint64_t bd =
              sm100::sdesc_k_plain(sm100::smem_u32(task.z & 1 ? a : a + tile_bytes), lead, 128);
          const int ksteps = min(box, len - off) / 16;
          for (int ks = 0; ks < ksteps; ++ks) {
            const uint64_t step = (uint64_t)(ks * (block_bytes >> 4));
            sm100::mma_bf16(acc_at, ad + step, bd + step, idesc, acc);
            acc = 1;
          }
          sm100::mma_commit(&empty[st]);
          if (++st == S) {
            st = 0;
            ph ^= 1;
          }
        }
      }
      sm100::mma_commit(&acc_full[buf]);
    }
    sm100::mma_commit(&done);
    if (!ok) atomicOr(&flags[2], 1);
  } else if (warp >= 2) {
    // epilogue: warp w reads TMEM lanes 32 (w mod 4) .. + 31 (= rows of the block)
    const int quad = warp & 3, m = 32 * quad + lane;
    const bool vec = K % 4 == 0;
    int q = 0;
    for (int t = t0; t < t1 && ok; ++t, ++q) {
      const int buf = q & 1;
      const int4 task = tasks[t];
      // a pair is one chain: the wait grows with its boxes (each within the limits above)
      const uint32_t limit = sm100::kSpinLimit + 256u * min((uint32_t)(task.z >> 1), 1u << 22);
      if (!sm100::mbar_wait(&acc_full[buf], (q >> 1) & 1, limit)) {
        ok = false;
        break;
      }
      sm100::tc_fence_after();
      float* out = G + (int64_t)task.w * K * K + (int64_t)m * K;
      if (32 * quad < K) {
        for (int c0 = 0; c0 < N; c0 += 16) {
          uint32_t v[16];
          sm100::tmem_ld16(tmem + (uint32_t)buf * 128u + ((uint32_t)(32 * quad) << 16) + (uint32_t)c0,
                           v);
          sm100::tmem_ld_wait();
          if (m < K && vec) {
#pragma unroll
            for (int j = 0; j < 16; j += 4)
              if (c0 + j < K)
                *reinterpret_cast<float4*>(out + c0 + j) =
                    make_float4(__uint_as_float(v[j]), __uint_as_float(v[j + 1]),
                                __uint_as_float(v[j + 2]), __uint_as_float(v[j + 3]));
          } else if (m < K) {
#pragma unroll
            for (int j = 0; j < 16; ++j)
              if (c0 + j < K) out[c0 + j] = __uint_as_float(v[j]);
          }
          __syncwarp();   // the next load is warp-aligned
        }
      }
      sm100::tc_fence_before();
      __syncwarp();
      if (lane == 0) sm100::mbar_arrive(&acc_empty[buf]);
    }
    if (!ok && lane == 0) atomicOr(&flags[2], 1);
  }
  __syncwarp();
  // every MMA has completed before TMEM is given back
  if (!sm100::mbar_wait(&done, 0) && threadIdx.x == 0) atomicOr(&flags[2], 1);
  sm100::tc_fence_before();
  __syncthreads();
  sm100::tc_fence_after();
  if (warp == 2) sm100::tmem_dealloc(tmem, 256);
}

// out[n] = Gram block (which[n].x: its index, < 0 a zero block; which[n].y: transposed)
__global__ void __launch_bounds__(256) k_gram_blocks(const int2* __restrict__ which, int K,
                                                     const float* __restrict__ G,
                                                     double* __restrict__ out) {
  const int2 q = which[blockIdx.x];
  const int e = blockIdx.y * 256 + threadIdx.x;
  if (e >= K * K) return;
  const int a = e / K, b = e - a * K;
  out[(int64_t)blockIdx.x * K * K + e] =
      q.x < 0 ? 0.0 : (double)G[(int64_t)q.x * K * K + (q.y ? b * K + a : e)];
}

}  // namespace

// Pairs (i <= j) with shared rows, the runs of each and the CTA that takes it
// (host), for the assembled system.
void gram_build_pairs(elmfb_ctx* h) {
  struct Run {
    int a, b, len;   // panel rows of i and j
  };
  struct Task {
    int4 t;
    int at;   // the pair's first cell
    int boxes;
  };
  // the entries of every subdomain, in cell order
  const int ne = (int)h->cover_sub.size();
  std::vector<int> off(h->n_sub + 1, 0), ent(ne);
  for (int e = 0; e < ne; ++e) off[h->cover_sub[e] + 1]++;
  for (int s = 0; s < h->n_sub; ++s) off[s + 1] += off[s];
  {
    std::vector<int> fill(off.begin(), off.end() - 1);
    for (int e = 0; e < ne; ++e) ent[fill[h->cover_sub[e]]++] = e;
  }
  h->gram_pair_ij.clear();
  std::vector<Task> tasks;
  std::vector<int4> runs;
  int64_t total = 0;
  // subdomain by subdomain, its pairs' runs gathered by the partner
  std::vector<int> slot(h->n_sub, -1), partners, first_cell;
  std::vector<std::vector<Run>> runs_of;
  for (int s1 = 0; s1 < h->n_sub; ++s1) {
    partners.clear();
    first_cell.clear();
    for (int q = off[s1]; q < off[s1 + 1]; ++q) {
      const int e1 = ent[q], c = h->entry_cell[e1];
      if (h->cell_count[c] == 0) continue;
      const int pad = h->cell_pstart[c + 1] - h->cell_pstart[c];
      const int a = (int)(h->panel_off[s1] + h->cover_start[e1]);
      for (int e2 = e1; e2 < h->cover_off[c + 1]; ++e2) {
        const int s2 = h->cover_sub[e2];
        const int b = (int)(h->panel_off[s2] + h->cover_start[e2]);
        if (slot[s2] < 0) {
          slot[s2] = (int)partners.size();
          partners.push_back(s2);
          first_cell.push_back(c);
          if (runs_of.size() < partners.size()) runs_of.emplace_back();
          runs_of[slot[s2]].clear();
        }
        auto& v = runs_of[slot[s2]];
        if (!v.empty() && v.back().a + v.back().len == a && v.back().b + v.back().len == b)
          v.back().len += pad;
        else
          v.push_back({a, b, pad});
      }
    }
    std::sort(partners.begin(), partners.end());
    for (int s2 : partners) {
      const int k = slot[s2], r0 = (int)runs.size();
      slot[s2] = -1;
      int boxes = 0;
      for (const Run& r : runs_of[k]) {
        runs.push_back(make_int4(r.a, r.b, r.len, 0));
        boxes += (int)ceil_div(r.len, gram_box_rows(h->K));
      }
      tasks.push_back({make_int4(r0, (int)runs.size(), 2 * boxes + (s1 == s2),
                                 (int)h->gram_pair_ij.size()),
                       first_cell[k], boxes});
      h->gram_pair_ij.push_back({s1, s2});
      total += boxes;
    }
  }
  int sms = 0;
  CUDA_CHECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->device));
  const int ctas = (int)std::min<size_t>(tasks.size(), sms);
  // A box costs its CTA about the same whether one tile or two are read for it, so
  // boxes are what is shared out (by tiles: 0.99 instead of 0.79 ms).  Pairs above an
  // eighth of a CTA's share first, the longest before the others (all in spatial
  // order: 0.97 ms); the rest in the order of their first cell.
  const int64_t large = total / std::max(ctas, 1) / 8;
  std::stable_sort(tasks.begin(), tasks.end(), [large](const Task& x, const Task& y) {
    const bool lx = x.boxes > large, ly = y.boxes > large;
    if (lx != ly) return lx;
    return lx ? x.boxes > y.boxes : x.at < y.at;
  });
  std::vector<int> owner(tasks.size()), task_off(ctas + 1, 0);
  {
    typedef std::pair<int64_t, int> Load;   // boxes so far, CTA
    std::priority_queue<Load, std::vector<Load>, std::greater<Load>> idle;
    for (int c = 0; c < ctas; ++c) idle.push({0, c});
    for (size_t k = 0; k < tasks.size(); ++k) {
      const Load l = idle.top();
      idle.pop();
      owner[k] = l.second;
      task_off[l.second + 1]++;
      idle.push({l.first + tasks[k].boxes + 8, l.second});   // 8: a task's own cost
    }
    for (int c = 0; c < ctas; ++c) task_off[c + 1] += task_off[c];
  }
  std::vector<int4> flat(tasks.size());
  {
    std::vector<int> fill(task_off.begin(), task_off.end() - 1);
    for (size_t k = 0; k < tasks.size(); ++k) flat[fill[owner[k]]++] = tasks[k].t;
  }
  h->d_gram_task_off.alloc(task_off.size() * sizeof(int), h->stream);
  CUDA_CHECK(cudaMemcpyAsync(h->d_gram_task_off.p, task_off.data(), task_off.size() * sizeof(int),
                             cudaMemcpyHostToDevice, h->stream));
  h->gram_ctas = ctas;
  h->n_gram_pairs = (int64_t)h->gram_pair_ij.size();
  auto up = [&](DevBuf& d, const std::vector<int4>& v) {
    d.alloc(std::max<size_t>(v.size(), 1) * sizeof(int4), h->stream);
    if (!v.empty())
      CUDA_CHECK(cudaMemcpyAsync(d.p, v.data(), v.size() * sizeof(int4), cudaMemcpyHostToDevice,
                                 h->stream));
  };
  up(h->d_gram_tasks, flat);
  up(h->d_gram_runs, runs);
}

void gram_compute(elmfb_ctx* h) {
  if (h->cfg.precision != ELMFB_MIXED)
    ELMFB_THROW(ELMFB_ERR_UNSUPPORTED, "tensor-core Gram blocks need ELMFB_MIXED precision");
  if (h->K > 128) ELMFB_THROW(ELMFB_ERR_UNSUPPORTED, "tensor-core Gram blocks need K <= 128");
  cudaStream_t st = h->stream;
  if (h->gram_pair_ij.empty()) gram_build_pairs(h);
  const int K = h->K;
  const int N = (K + 15) & ~15;
  h->d_gram.alloc(std::max<int64_t>(h->n_gram_pairs, 1) * K * K * sizeof(float), st);
  ensure_dyn_smem((const void*)k_gram_tc, kGramSmem);
  CUDA_CHECK(cudaMemsetAsync(h->d_flags.p, 0, 16 * sizeof(int), st));
  stage_begin(h, 3);
  // algorithmic work: 2 K^2 flops per shared row per pair; bytes: BF16 rows read once
  prof_begin(h, KID_GRAM_TC, (double)h->NPR * K * 2.0 + (double)h->n_gram_pairs * K * K * 4.0);
  if (h->gram_ctas > 0) {
    const int S = (int)std::min<size_t>(kMaxGramStages, kGramRing / (2 * gram_tile_bytes(K)));
    k_gram_tc<<<(unsigned)h->gram_ctas, kGramThreads, kGramSmem, st>>>(
        h->d_pt.as<uint8_t>(), h->d_gram_tasks.as<int4>(), h->d_gram_task_off.as<int>(),
        h->d_gram_runs.as<int4>(), K, N, S, h->d_gram.as<float>(), h->d_flags.as<int>());
  }
  prof_end(h, KID_GRAM_TC);
  check_launch("k_gram_tc");
  count_launch(h);
  stage_end(h, 3);
  int flags[4];
  CUDA_CHECK(cudaMemcpyAsync(flags, h->d_flags.p, 4 * sizeof(int), cudaMemcpyDeviceToHost, st));
  stream_sync(h);
  if (flags[2]) ELMFB_THROW(ELMFB_ERR_TIMEOUT, "tensor-core Gram: a pipeline wait timed out");
  h->have_gram = true;
}

extern "C" {

int elmfb_compute_gram(elmfb_t h) {
  if (!h) return ELMFB_ERR_INVALID_ARG;
  try {
    CUDA_CHECK(cudaSetDevice(h->device));
    if (!h->assembled) ELMFB_THROW(ELMFB_ERR_STATE, "compute_gram before assemble");
    gram_compute(h);
    return ELMFB_OK;
  } catch (const elmfb_error& e) {
    h->err = e.msg;
    return e.code;
  } catch (const std::bad_alloc&) {
    h->err = "host allocation failed";
    return ELMFB_ERR_OOM;
  } catch (const std::exception& e) {
    h->err = e.what();
    return ELMFB_ERR_CUDA;
  }
}

int elmfb_get_gram(elmfb_t h, int64_t n, const int* ij, double* out) {
  if (!h) return ELMFB_ERR_INVALID_ARG;
  try {
    CUDA_CHECK(cudaSetDevice(h->device));
    if (!h->have_gram) ELMFB_THROW(ELMFB_ERR_STATE, "get_gram before compute_gram");
    if (n < 0 || (n > 0 && (!ij || !out))) ELMFB_THROW(ELMFB_ERR_INVALID_ARG, "bad arguments");
    const int K = h->K;
    std::vector<int> hij(2 * n);
    CUDA_CHECK(cudaMemcpy(hij.data(), ij, 2 * n * sizeof(int), cudaMemcpyDefault));
    if (n == 0) return ELMFB_OK;
    std::vector<int2> which(n);
    for (int64_t q = 0; q < n; ++q) {
      int i = hij[2 * q], j = hij[2 * q + 1];
      const bool tr = i > j;
      if (tr) std::swap(i, j);
      auto it = std::lower_bound(h->gram_pair_ij.begin(), h->gram_pair_ij.end(),
                                 std::make_pair(i, j));
      const bool found = it != h->gram_pair_ij.end() && *it == std::make_pair(i, j);
      which[q] = make_int2(found ? (int)(it - h->gram_pair_ij.begin()) : -1, tr);
    }
    // In place in device memory, else through a staging buffer, a slice at a time; on
    // the legacy stream, as a plain copy to `out` would be, so that work on `out` that
    // is pending there or on blocking streams comes first (the blocks themselves were
    // complete when compute_gram returned).
    cudaStream_t st = cudaStreamLegacy;
    const int64_t KK = (int64_t)K * K;
    const bool direct = usable_in_place(h, out, sizeof(double));
    const int64_t slice = std::min<int64_t>(
        n, direct ? int64_t(1) << 24 : std::max<int64_t>(1, kGramStaging / (KK * sizeof(double))));
    DevBuf dw, dout;
    dw.alloc(slice * sizeof(int2), st);
    if (!direct) dout.alloc(slice * KK * sizeof(double), st);
    for (int64_t q = 0; q < n; q += slice) {
      const int64_t c = std::min(slice, n - q);
      double* const o = direct ? out + q * KK : dout.as<double>();
      CUDA_CHECK(cudaMemcpyAsync(dw.p, which.data() + q, c * sizeof(int2), cudaMemcpyHostToDevice,
                                 st));
      k_gram_blocks<<<dim3((unsigned)c, (unsigned)ceil_div(KK, 256)), 256, 0, st>>>(
          dw.as<int2>(), K, h->d_gram.as<float>(), o);
      check_launch("k_gram_blocks");
      count_launch(h);
      if (!direct)
        CUDA_CHECK(cudaMemcpyAsync(out + q * KK, o, c * KK * sizeof(double), cudaMemcpyDefault, st));
    }
    CUDA_CHECK(cudaStreamSynchronize(st));
    return ELMFB_OK;
  } catch (const elmfb_error& e) {
    h->err = e.msg;
    return e.code;
  } catch (const std::bad_alloc&) {
    h->err = "host allocation failed";
    return ELMFB_ERR_OOM;
  } catch (const std::exception& e) {
    h->err = e.what();
    return ELMFB_ERR_CUDA;
  }
}

}  // extern "C"
