// Internal hooks between the handle code and the request server (not part of the ABI).
#pragma once
#include <cuda_runtime.h>

#include "../../include/me.h"

// Enqueue, on the handle's stream, a copy of the last call's rescue count to `dst`
// (host-pinned); returns ME_OK or an error code.
int me_internal_rescued_async(me_handle* h, int* dst);
// Launches of one batch whose size is read on the device (*d_n <= cap; momenta with
// stride cap, weights optional): the main kernel, the float64 rescue of the flagged
// points (mixed precision, subtracted real) and the reduction, on the handle's stream.
// Allocates nothing and never synchronises, so the sequence can be captured in a CUDA
// graph and replayed for any batch size up to cap.  me_internal_prepare_counted (outside
// any capture, after one ordinary call of the kind) sizes the handle's scratch for cap.
int me_internal_prepare_counted(me_handle* h, int me_kind, int64_t cap);
int me_internal_launch_counted(me_handle* h, int me_kind, const double* d_p, const double* d_w, int64_t cap,
                               const int* d_n, double* d_out);
// Whether a subtracted-real call of n points runs the per-term queues (1), the masked evaluation (0),
// or is not defined (-1); a rule on the arguments alone.
extern "C" int me_internal_term_queues(const char* process, const me_params* params, int64_t n);
// Failure injection on the host, for tests: the calling thread's next evaluation of a handle
// reports a launch failure in place of its main kernel (stage 1), its float64 rescue (2) or its
// reduction (3), with what comes before launched and nothing after.
extern "C" void me_internal_fail_stage(int stage);
// Final-state masses of the handle's process (outgoing legs in order; at most 4), their
// number, and the handle's stream.
int me_internal_final_masses(me_handle* h, double* masses, int* n_out, cudaStream_t* stream);
// A workspace for one call: device memory of at least `bytes` (stream-ordered on `st`) and 64 B of
// mapped host memory with its device address.  Each call takes its own, so that several
// threads can use one handle, and gives it back once `st` has finished with it; the handle keeps
// a few for later calls and releases the others.
struct Workspace {
  void* dev;
  size_t bytes;
  void* host;
  void* host_dev;
};
int me_internal_workspace_take(me_handle* h, size_t bytes, cudaStream_t st, Workspace* out);
void me_internal_workspace_give(me_handle* h, Workspace w, cudaStream_t st);
// Process id (index into the library's process table) of a name, or -1.
int me_internal_process_id(const char* name);
// Process id of a handle, or -1 for NULL.
int me_internal_handle_process(const me_handle* h);
// Record the thread-local message returned by me_last_error(); returns `code`.
int me_internal_fail(int code, const char* msg);

namespace me {
struct ColourTables;
struct KParams;
}  // namespace me
// Fill host colour tables (the same construction as the per-device set-up).
int me_internal_build_tables(me::ColourTables* tab);
// Validate parameters and fill kernel parameters for a process (tables pointer unset).
int me_internal_kparams(const char* process, const me_params* params, me::KParams* kp, int* pid);
// The same with the device-resident tables of params->device set up and filled in.
int me_internal_device_kparams(const char* process, const me_params* params, me::KParams* kp, int* pid);
// Whether a buffer of CUDA memory type `mem_type` on device `mem_device` can be handed to
// a kernel on `want_device` without peer access (1) or not (0); exported with C linkage.
extern "C" int me_internal_buffer_usable(int mem_type, int mem_device, int want_device);
