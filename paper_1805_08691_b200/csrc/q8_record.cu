// Recording of library calls as a CUDA graph on streams of the library's own.
//
// A host that enqueues the same calls over and over pays more for enqueueing a short kernel than the GPU pays for running
// it.  The streams of a recording are created for it and belong to nobody else: a framework hands out streams from a pool,
// and work that another thread enqueues on a stream which happens to be recording would end up in the graph instead of on
// the GPU.  Relaxed capture mode: kernels may be loaded on first use while they are recorded, and no other thread's calls
// are restricted.
#include "q8_internal.h"

namespace q8 {
namespace {

void destroy_streams(int n, void** streams) {
  for (int i = 0; i < n; ++i) {
    if (streams[i]) cudaStreamDestroy(as_stream(streams[i]));
    streams[i] = nullptr;
  }
}

}  // namespace
}  // namespace q8

using namespace q8;

extern "C" {

int q8_record_begin(int n_streams, void** streams) {
  clear_error();
  if (!streams || n_streams < 1) return fail(Q8_ERR_INVALID_ARG, "q8_record_begin: null pointer or no stream");
  for (int i = 0; i < n_streams; ++i) streams[i] = nullptr;
  int rc = Q8_OK;
  for (int i = 0; i < n_streams && rc == Q8_OK; ++i) {
    cudaStream_t s = nullptr;
    rc = check_cuda(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking), "q8_record_begin: create stream");
    streams[i] = s;
  }
  if (rc == Q8_OK) rc = check_cuda(cudaStreamBeginCapture(as_stream(streams[0]), cudaStreamCaptureModeRelaxed), "q8_record_begin: begin capture");
  if (rc != Q8_OK) destroy_streams(n_streams, streams);
  return rc;
}

int q8_record_end(int n_streams, void** streams, void** graph) {
  clear_error();
  if (!streams || n_streams < 1 || !streams[0]) return fail(Q8_ERR_INVALID_ARG, "q8_record_end: null pointer or no stream");
  if (graph) *graph = nullptr;
  cudaGraph_t recorded = nullptr;
  cudaGraphExec_t exec = nullptr;
  int rc = check_cuda(cudaStreamEndCapture(as_stream(streams[0]), &recorded), "q8_record_end: end capture");
  if (rc == Q8_OK && graph) rc = check_cuda(cudaGraphInstantiate(&exec, recorded, 0), "q8_record_end: instantiate");
  // the launch data goes to the device now, not with the first replay
  if (exec) rc = check_cuda(cudaGraphUpload(exec, as_stream(streams[0])), "q8_record_end: upload");
  if (recorded) cudaGraphDestroy(recorded);
  destroy_streams(n_streams, streams);
  if (rc == Q8_OK && graph) *graph = exec;
  else if (exec) cudaGraphExecDestroy(exec);
  if (rc != Q8_OK) cudaGetLastError();  // a recording that cannot be ended leaves its error to the next launch otherwise
  return graph ? rc : Q8_OK;
}

int q8_record_replay(void* graph, void* stream) {
  clear_error();
  if (!graph) return fail(Q8_ERR_INVALID_ARG, "q8_record_replay: null pointer");
  return check_cuda(cudaGraphLaunch(static_cast<cudaGraphExec_t>(graph), as_stream(stream)), "q8_record_replay");
}

int q8_record_free(void* graph) {
  clear_error();
  if (!graph) return Q8_OK;
  return check_cuda(cudaGraphExecDestroy(static_cast<cudaGraphExec_t>(graph)), "q8_record_free");
}

}  // extern "C"
