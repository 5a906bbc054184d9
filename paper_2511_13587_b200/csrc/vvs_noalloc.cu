// vvs_decide_noalloc: the decision stage (acceptance test, accepted prefix, residual / bonus
// sample) for callers that must not allocate device memory.  The same kernel as vvs_decide, which keeps
// everything between its steps in registers and shared memory; only the status word lives here.
#include <mutex>

#include "vvs_internal.cuh"

using namespace vvs;

namespace {

constexpr int kMaxImages = VVS_NOALLOC_MAX_IMAGES;
constexpr int kMaxDrafts = VVS_NOALLOC_MAX_DRAFTS;
constexpr int kMaxNbrK = VVS_NOALLOC_MAX_NBR_K;
constexpr int kMaxVocab = VVS_NOALLOC_MAX_VOCAB;

// Status word of callers that pass none: the decision kernel needs no other scratch.  Resident on every GPU that
// loads this library.  In host code this name is only a stand-in for the symbol, not a device address: the
// address the kernel gets comes from cudaGetSymbolAddress below.
static __device__ int32_t g_noalloc_status;

constexpr int kMaxDevices = 64;
std::mutex g_mu;
int32_t* g_status_addr[kMaxDevices] = {};  // device address of the word, per device ordinal

// Once per device, with that device current: resolve the device address of the word.
int status_for_current_device(int32_t** out) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return VVS_ERR_CUDA;
  std::lock_guard<std::mutex> lock(g_mu);
  if (!g_status_addr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc_status) != cudaSuccess || !p) {
      cudaGetLastError();
      return VVS_ERR_CUDA;
    }
    g_status_addr[dev] = static_cast<int32_t*>(p);
  }
  *out = g_status_addr[dev];
  return VVS_OK;
}

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

}  // namespace

extern "C" int vvs_decide_noalloc(const float* target_probs, int32_t vocab, int32_t vocab_offset,
                                  int32_t n_rows_per_seq, int32_t first_row, const int32_t* drafts,
                                  const int32_t* nbr_row_ptr, const int32_t* nbr_col,
                                  const vvs_verify_args* a, const vvs_verify_out* o,
                                  int32_t* status_bits, void* stream) {
  if (!target_probs || !a || !o) return VVS_ERR_INVALID_ARG;
  if (!a->uniforms || !o->accept_len || !o->next_token) return VVS_ERR_INVALID_ARG;
  if (a->n_cfg != 1 || a->n_images < 1 || a->n_draft_max < 0 || n_rows_per_seq < 1) return VVS_ERR_SHAPE;
  // documented capacity
  if (a->n_images > kMaxImages || a->n_draft_max > kMaxDrafts || vocab < 1 || vocab > kMaxVocab)
    return VVS_ERR_SHAPE;
  if (vocab_offset < 0 || first_row < 0 || first_row + a->n_draft_max > n_rows_per_seq) return VVS_ERR_SHAPE;
  if (a->n_draft_max > 0 && (!drafts || !a->draft_probs)) return VVS_ERR_INVALID_ARG;
  if (a->mode != VVS_MODE_STRICT && a->mode != VVS_MODE_RELAXED) return VVS_ERR_INVALID_ARG;
  if (a->mode == VVS_MODE_RELAXED) {
    if (a->nbr_k < 1 || a->nbr_k > kMaxNbrK) return VVS_ERR_SHAPE;
    if (!(a->delta >= 0.f)) return VVS_ERR_INVALID_ARG;
    if (a->nbr_k > 1 && (!nbr_row_ptr || !nbr_col)) return VVS_ERR_NOT_BOUND;
  }
  if (o->new_len || o->n_commit || o->hidden || o->target_probs) return VVS_ERR_INVALID_ARG;
  // chains only: a candidate tree needs the walk's float64 scratch rows
  if (a->tree_parent || o->accept_path) return VVS_ERR_INVALID_ARG;
  if (a->adjusted_residual != 0) return VVS_ERR_INVALID_ARG;   // needs a writable copy of the sampled row
  if (!aligned16(target_probs) || !aligned16(a->draft_probs)) return VVS_ERR_ALIGN;

  Workspace ws;  // only the status word is touched
  ws.status = status_bits;
  if (!status_bits) {
    const int rc = status_for_current_device(&ws.status);
    if (rc != VVS_OK) return rc;
  }

  DecideParams p{};
  p.n_images = a->n_images; p.n_cfg = 1; p.rows_per_seq = n_rows_per_seq; p.first_row = first_row;
  p.n_draft_max = a->n_draft_max; p.vocab = vocab; p.vocab_offset = vocab_offset;
  p.mode = a->mode; p.nbr_k = a->mode == VVS_MODE_RELAXED ? a->nbr_k : 1; p.kmax = kMaxNbrK;
  p.delta = a->delta;
  p.drafts = drafts; p.drafts_ld = a->n_draft_max; p.n_draft = a->n_draft;
  p.draft_probs = a->draft_probs; p.uniforms = a->uniforms;
  p.row_ptr = nbr_row_ptr; p.col = nbr_col;
  p.direct_probs = target_probs;
  p.n_forced = 1;
  p.accept_len = o->accept_len; p.next_token = o->next_token;
  p.accept_mask = o->accept_mask; p.margins = o->margins;

  return launch_decide(target_probs, false, 0, ws, p, true, static_cast<cudaStream_t>(stream));
}
