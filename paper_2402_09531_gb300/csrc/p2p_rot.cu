// Launches of the float32 near field that evaluates each unordered pair once
// (p2p_rot.cuh), for one tree and for a batch's right-hand-side class.
#include <algorithm>
#include <atomic>
#include <vector>

#include "p2p_rot.cuh"

namespace dw {

namespace {

using namespace rot;

constexpr size_t kRotMaxBytes = size_t(8) << 30;   // partial sums

template <int D, int RC, int KER>
__global__ void __launch_bounds__(kRotThreads, RC > 4 ? 3 : 4) k_near_rot(const RotArgs a) {
  extern __shared__ __align__(16) float rsm[];
  rot_chunk<D, RC, KER>(a, static_cast<int>(blockIdx.x), rsm);
}

template <int D, int RC, int KER>
void rot_launch(const RotArgs& a, int chunks, cudaStream_t s) {
  constexpr size_t most = rot_smem<D, RC>(kRotMaxLeaf);
  if (most > 48 * 1024) {
    static std::atomic<uint64_t> done{0};
    const uint64_t bit = device_bit();
    if (!(done.load() & bit)) {
      DW_CUDA(cudaFuncSetAttribute(k_near_rot<D, RC, KER>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   static_cast<int>(most)));
      done.fetch_or(bit);
    }
  }
  k_near_rot<D, RC, KER><<<chunks, kRotThreads, rot_smem<D, RC>(a.ld), s>>>(a);
}

template <int D, int RC>
void rot_kernel(int kernel, const RotArgs& a, int chunks, cudaStream_t s) {
  if (kernel == DWFMM_K_EXP) rot_launch<D, RC, DWFMM_K_EXP>(a, chunks, s);
  else if (kernel == DWFMM_K_MATERN32) rot_launch<D, RC, DWFMM_K_MATERN32>(a, chunks, s);
  else rot_launch<D, RC, DWFMM_K_GAUSS>(a, chunks, s);
}

template <int D>
void rot_rc(int kernel, int RC, const RotArgs& a, int chunks, cudaStream_t s) {
  if (RC <= 1) rot_kernel<D, 1>(kernel, a, chunks, s);
  else if (RC <= 4) rot_kernel<D, 4>(kernel, a, chunks, s);
  else rot_kernel<D, 8>(kernel, a, chunks, s);
}

void rot_dispatch(int D, int kernel, int RC, const RotArgs& a, int chunks, cudaStream_t s) {
  switch (D) {
    case 4: rot_rc<4>(kernel, RC, a, chunks, s); break;
    case 8: rot_rc<8>(kernel, RC, a, chunks, s); break;
    case 10: rot_rc<10>(kernel, RC, a, chunks, s); break;
    case 12: rot_rc<12>(kernel, RC, a, chunks, s); break;
    case 16: rot_rc<16>(kernel, RC, a, chunks, s); break;
    default: rot_rc<20>(kernel, RC, a, chunks, s); break;
  }
}

}  // namespace

void launch_rot(int D, int kernel, int RC, const RotArgs& a, int chunks, cudaStream_t s) {
  if (chunks > 0) rot_dispatch(D, kernel, RC, a, chunks, s);
}

size_t persist_rot_bytes(int D, int RC, int ld) {
  switch (D) {
#define DW_ROT_BYTES(DV) case DV: return RC <= 1 ? rot_smem<DV, 1>(ld) : RC <= 4 ? rot_smem<DV, 4>(ld) : rot_smem<DV, 8>(ld);
    DW_ROT_BYTES(4)
    DW_ROT_BYTES(8)
    DW_ROT_BYTES(10)
    DW_ROT_BYTES(12)
    DW_ROT_BYTES(16)
    DW_ROT_BYTES(20)
#undef DW_ROT_BYTES
  }
  return 0;
}

int rot_sources_per_chunk() { return kRotPer; }
bool rot_fits(int ld, int least, int rc) { return ld <= kRotMaxLeaf && least >= kRotMinLeaf && rc <= kRotMaxRc; }

// Chunks of `per` sources of every leaf's upper row; false when a leaf has
// fewer than `least` sites.
bool row_chunks(Plan& P, int per, int least, RowChunks& out) {
  if (!P.sym_ok || static_cast<int>(P.h_upcount.size()) != P.L) return false;
  int cmin = 1 << 30, cmax = 0;
  for (int l = 0; l < P.L; ++l) {
    cmin = std::min(cmin, P.h_count[P.L - 1 + l]);
    cmax = std::max(cmax, P.h_count[P.L - 1 + l]);
  }
  if (cmin < least) return false;
  std::vector<int32_t> ptr(P.L + 1, 0), ct;
  for (int t = 0; t < P.L; ++t) {
    const int n = ceil_div(static_cast<int64_t>(P.h_upcount[t]) * cmax, per);
    ptr[t + 1] = ptr[t] + n;
    ct.insert(ct.end(), n, t);
  }
  out.n = ptr[P.L];
  out.cmax = cmax;
  out.t.alloc(ct.size());
  out.ptr.alloc(ptr.size());
  DW_CUDA(cudaMemcpyAsync(out.t.p, ct.data(), ct.size() * sizeof(int32_t), cudaMemcpyHostToDevice, P.stream));
  DW_CUDA(cudaMemcpyAsync(out.ptr.p, ptr.data(), ptr.size() * sizeof(int32_t), cudaMemcpyHostToDevice, P.stream));
  DW_CUDA(cudaStreamSynchronize(P.stream));
  return true;
}

// Whether the near field of Rc right-hand sides takes this form; builds the
// tree's chunks on first use.  Called before the side stream forks.  Above 8
// right-hand sides the sums of both sides leave the registers (and MIXED plans
// have the tensor cores); leaves below 32 sites would make lanes of a turn
// share a target; partial sums beyond 8 GB are not worth their traffic, and where
// there is no memory for them the list kernel needs none.
bool rot_ready(Plan& P, int Rc) {
  if (sum_padded_dim(P.d) < 0 || !rot_fits(P.m_pad, kRotMinLeaf, sum_padded_rc(Rc))) return false;
  if (P.rot_state < 0 && capturing(P.stream)) return false;   // the chunks are built outside a capture
  if (P.rot_state < 0) P.rot_state = row_chunks(P, kRotPer, kRotMinLeaf, P.rot) ? 1 : 0;
  if (P.rot_state == 0) return false;
  const size_t row = round_up(P.rot.cmax, 8);
  const size_t most = kRotMaxBytes / ((static_cast<size_t>(P.rot.n) + P.sym_nup) * row * sizeof(float));
  if (most < static_cast<size_t>(Rc)) return false;
  const size_t cols = P.work_cols(Rc, sum_padded_rc(Rc), most);
  return P.grow(P.rot_pf, P.rot.n * row * cols) && P.grow(P.rot_pt, P.sym_nup * row * cols);
}

// pts: scaled blocks of the leaves; charges in P.xq32.
void near_rot(Plan& P, int D, int Rc, cudaStream_t s) {
  RotArgs a{};
  a.pts = P.d_ptsk.p;
  a.q = P.xq32.p;
  a.count = P.d_count.p + P.L - 1;
  a.chunk_t = P.rot.t.p;
  a.chunk_ptr = P.rot.ptr.p;
  a.uprow = P.sym_uprow.p;
  a.up_s = P.sym_s.p;
  a.ld = P.m_pad;
  a.Rc = Rc;
  a.ldp = round_up(P.rot.cmax, 8);
  a.cmax = P.rot.cmax;
  a.pf = P.rot_pf.p;
  a.pt = P.rot_pt.p;
  rot_dispatch(D, P.kernel, sum_padded_rc(Rc), a, P.rot.n, s);
}

}  // namespace dw
