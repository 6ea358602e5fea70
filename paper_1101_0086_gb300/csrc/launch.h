// Host-side launchers of the kernels in kernels.cuh (one translation unit
// per kernel family and precision, compiled in parallel).
#pragma once

#include <atomic>

#include "kernels.cuh"

namespace mpa {

// Kernels launched by this library since load.
extern std::atomic<long long> g_launches;

// Host-side fault injection (mpa_debug_fail_launch): when armed, the launch
// gate of the n-th kernel launch from now returns the chosen error instead
// of launching, so the error paths of every entry point can be exercised
// without making a GPU fault.  Every launcher calls it before its launch.
extern std::atomic<long long> g_fail_countdown;  // < 0: disarmed
extern std::atomic<int> g_fail_code;
inline cudaError_t launch_gate() {
    if (g_fail_countdown.load(std::memory_order_relaxed) < 0) return cudaSuccess;
    const long long left = g_fail_countdown.fetch_sub(1, std::memory_order_acq_rel);
    if (left == 0) return static_cast<cudaError_t>(g_fail_code.load(std::memory_order_relaxed));
    if (left < 0) g_fail_countdown.store(-1, std::memory_order_relaxed);
    return cudaSuccess;
}

// One-time kernel attribute setup per device: cudaFuncSetAttribute applies
// to the current device only, so each launcher keeps one bit per device
// (devices 0..63; any higher device sets the attributes on every launch).
// Setting an attribute twice is harmless, so two threads racing on the first
// launch of a device need no lock.
struct AttrOnce {
    std::atomic<unsigned long long> mask{0};
};
template <class F> inline cudaError_t attrs_once(AttrOnce& once, F&& set) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = dev >= 0 && dev < 64 ? 1ull << dev : 0ull;
    if (bit && (once.mask.load(std::memory_order_acquire) & bit)) return cudaSuccess;
    e = set();
    if (e == cudaSuccess && bit) once.mask.fetch_or(bit, std::memory_order_acq_rel);
    return e;
}

// SMs of the current device, asked for once a device (devices 0..63).
inline cudaError_t sm_count(int* sms) {
    static std::atomic<int> known[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const bool keep = dev >= 0 && dev < 64;
    if (keep && (*sms = known[dev].load(std::memory_order_relaxed)) > 0) return cudaSuccess;
    e = cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess && keep) known[dev].store(*sms, std::memory_order_relaxed);
    return e;
}
// Whether `blocks` blocks fill `sms` SMs twice over.
inline bool fills_twice(long long blocks, int sms) { return blocks >= 2ll * sms; }

// Launch of a kernel that calls pdl_wait() before its first global access
// (device.cuh): its launch and preparation overlap the end of the kernel
// before it in the stream.  Split step of 2^14 modes (two kernels whose tables
// and launches took longer than their transforms) 13.9 -> 6.2 us, one span of
// a 2^16 link 3.94 -> 3.66 ms.  early = false: an ordinary launch.
template <class... P, class... A>
inline cudaError_t launch_pdl(bool early, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                              A... args) {
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = st;
    cudaLaunchAttribute a{};
    a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &a;
    c.numAttrs = early ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
    if (e != cudaSuccess) cudaGetLastError();  // returned here, not left for a later check of another call's
    return e;
}
// Whether a level's kernel of `blocks` blocks starts early: a grid that does
// not fill the SMs twice over would be packed onto the first ones that fall
// free.  Two intervals of three levels, ordinary / early, us: 2^13 x 143 nodes
// (143 blocks of transforms, 256 of the scan) 185 / 201, one interval of 2^12 x
// 801 (401, 128) 168 / 192, 2^13 x 801 (801, 256) 258 / 269.  At 2^12 x 143 (143
// blocks of 256 threads, 128) early is the faster, 141 / 122; the line lies
// where most grids gain.
inline bool pdl_fills(long long blocks) {
    int sms = 0;
    return sm_count(&sms) == cudaSuccess && fills_twice(blocks, sms);
}
// Whether two CTAs with `smem` bytes of shared memory each fit an SM (228 KB, 1
// KB of them reserved for each).
constexpr bool pair_fits(size_t smem) { return 2 * (smem + 1024) <= 228 * 1024; }
// Whether an FP64 column or row pass of a level starts early.  Where two of its
// CTAs fit an SM (`pair`) and it has at most one for each SM, an early start
// packs them in pairs onto half of the SMs, and an FP64 CTA takes as long as the
// SM's FP64 pipe has work.  A level of 143 nodes, early / ordinary: 2^12 (143
// blocks a column pass) 415 / 293 us, 2^11 with columns of 64 (72 blocks) 268 /
// 236.  CTAs that get an SM each in any case lose only the overlap by an ordinary
// launch (2^10, columns of 32: 237 / 315; 2^13, 286 blocks: 560 / 569), and the
// overlap is worth more than the packing of a few (2^10 with columns of 64, 36
// blocks: 210 / 224).
inline bool pdl_level64(bool pair, long long blocks, int sms) { return !pair || 4 * blocks <= sms || blocks > sms; }
// Whether a pass over a single field of n samples starts early.  FP64 passes of
// 2^16 .. 2^18 samples, bound by the schedulers they spread over, would be
// packed too: us a split step, early / ordinary: 2^14 27 / 46, 2^15 31 / 43,
// 2^16 86 / 42, 2^17 157 / 68, 2^18 189 / 123, 2^19 230 / 237, 2^20 412 / 419;
// FP32: 2^14 6.2 / 13.9, 2^18 12.9 / 13.8, 2^20 23.3 / 23.2, 2^22 66 / 71.  The
// two passes of a transform of 2^19 samples are packed as well: 127 / 99 (2^20
// 173 / 180).
template <typename T> inline bool pdl_field(long long n, bool transform = false) {
    return sizeof(T) == 4 || n <= (1ll << 15) || n > (1ll << (transform ? 19 : 18));
}

// Optional CUDA-event timing of every launch, by kernel kind (off by
// default; enabled through mpa_profile).
enum {
    PK_KC_MPA_PRE = 0, PK_KC_MPA_POST, PK_KC_SS, PK_KC_FFT, PK_KR_MPA, PK_KR_SS, PK_KR_FFT, PK_SCAN, PK_AUX,
    PK_KCW, PK_KC_ADJ, PK_KR_ADJ, PK_ADJ_AUX, PK_KN, PK_COUNT
};
extern std::atomic<bool> g_prof_on;
void prof_begin(cudaStream_t st);
void prof_end(int kind, cudaStream_t st, double bytes);
// levels: a pass of the MPA levels (its transforms count with the MPA passes)
int prof_kc_kind(int mode, bool levels);
// Per-call timer of the entry points (mpa_last_timing): while profiling is
// on, the outermost timed entry point of a thread records a CUDA event on
// its stream at construction and at destruction (not on a capturing stream).
class CallTimer {
  public:
    CallTimer(const char* name, cudaStream_t st);
    ~CallTimer();
    CallTimer(const CallTimer&) = delete;
    CallTimer& operator=(const CallTimer&) = delete;

  private:
    const char* name_;
    cudaStream_t st_;
    cudaEvent_t a_ = nullptr;
};
void call_timing_reset();
// the most recent timed call: *have = false if there is none
cudaError_t call_timing_read(double* ms, const char** entry, bool* have);
int prof_kr_kind(int mode);
cudaError_t prof_read(int kind, double* ms, long long* n, double* bytes);
void prof_reset();

// Column/row lengths supported by the column pass (2^4..2^11) and the row
// pass (2^4..2^14 FP32, 2^4..2^13 FP64).
constexpr int KC_LOG_MIN = 4, KC_LOG_MAX = 11;
constexpr int KR_LOG_MIN = 4;
template <typename T> constexpr int kr_log_max() { return sizeof(T) == 4 ? 14 : 13; }

template <typename T> cudaError_t kc_launch(int mode, int logL, const KCParams<T>& p, cudaStream_t st);
template <typename T> cudaError_t kr_launch(int mode, int logL, const KRParams<T>& p, cudaStream_t st);
// whether kr_launch<float> takes the staged persistent row pass (krs.cuh)
bool kr_staged(int mode, int logL, const KRParams<float>& p);
// whether kc_launch<float> takes the staged persistent column pass (kcs.cuh)
bool kc_staged(int mode, int logL, const KCParams<float>& p);
// log2 of the columns per tile of the staged column pass for 2^logL-point
// columns (the tile layout's G), or -1 where there is none
int kcs_tile_log_cols(int logL);
// On-chip whole node transform for N = 2^logL, 2^8 <= N <= 2^kn_log_max:
// one CTA per node up to 2^14 (FP32) / 2^13 (FP64), a cluster of 2 or 4 CTAs
// over distributed shared memory for FP32 2^15 and 2^16 (knc_launch).
constexpr int KN_LOG_MIN = 8;
template <typename T> constexpr int kn_log_max() { return sizeof(T) == 4 ? 16 : 13; }
template <typename T> cudaError_t kn_launch(int logL, const KNParams<T>& p, cudaStream_t st);
cudaError_t knc_launch(int logL, const KNParams<float>& p, cudaStream_t st);
// Rows (nodes) per tile and threads per CTA of the FP32 on-chip transform
// for N = 2^logL <= 2^14 (KNGeom<float, N>: tiles of 8192 elements, 32 per thread).
#define KN_TILE_ROWS(logL) ((logL) >= 13 ? 1ll : (8192ll >> (logL)))
#define KN_THREADS(logL) ((logL) >= 14 ? 512ll : 256ll)
// Persistent batch kernel (kp.cuh): FP32, N = 2^logL <= 2^14, and its queue reset.
struct KPParams;
cudaError_t kp_launch(int logL, const KPParams& p, cudaStream_t st);
cudaError_t kp_init_launch(unsigned int* q_seq, unsigned int q_cap, unsigned int* ctr, int n_ctr, cudaStream_t st);
template <typename T> cudaError_t scan_launch(const ScanParams<T>& p, int links, cudaStream_t st);
template <typename T> cudaError_t transpose_launch(const cx<T>* in, cx<T>* out, long long R, long long C, cudaStream_t st);
template <typename T> cudaError_t to_state_launch(const cx<T>* in, double2* state, cx<T>* copy, long long N, cudaStream_t st);
template <typename T> cudaError_t from_state_launch(const double2* state, cx<T>* out, long long N, cudaStream_t st);

// Wavefront column pass (FP32): columns per tile for column length 2^logL,
// the launch, and the step-7 kernel that follows a wavefront interval.
int kcw_tile_cols(int logL);
cudaError_t kcw_launch(int logL, const KCWParams& p, cudaStream_t st);
cudaError_t reconstruct_launch(double2* state, float2* psi0c, const double2* D, const NodeC& nodeM, double gain,
                               long long N, unsigned int* err, double2* out, cudaStream_t st);

// Grid of a column pass over ncols columns of column length L.
template <typename T> long long kc_blocks(int logL, long long ncols);
template <typename T> long long kr_blocks(int logL, long long nrows);

}  // namespace mpa
