// Replayable launch sequences (CUDA graphs) for programs that issue the same calls again and again.
#include "ebs_internal.cuh"

using namespace ebs;

extern "C" {

int ebs_graph_begin(void** capture_stream) {
    if (!capture_stream) return EBS_ERR_INVALID_ARG;
    // a stream of its own: the legacy default stream cannot be captured, and the caller's stream keeps running meanwhile
    cudaStream_t st = nullptr;
    if (check_cuda(cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking))) return EBS_ERR_CUDA;
    if (check_cuda(cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal))) {
        cudaStreamDestroy(st);
        return EBS_ERR_CUDA;
    }
    *capture_stream = st;
    return EBS_OK;
}

int ebs_graph_end(void* capture_stream, void** graph_exec) {
    if (!capture_stream) return EBS_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(capture_stream);
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    int rc = check_cuda(cudaStreamEndCapture(st, &graph));
    if (!rc && graph_exec) rc = check_cuda(cudaGraphInstantiate(&exec, graph, 0));
    if (graph) cudaGraphDestroy(graph);
    cudaStreamDestroy(st);
    if (!rc && graph_exec) *graph_exec = exec;
    return rc;
}

int ebs_graph_launch(void* graph_exec, void* stream) {
    if (!graph_exec) return EBS_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    if (check_cuda(cudaStreamIsCapturing(st, &status))) return EBS_ERR_CUDA;
    if (status != cudaStreamCaptureStatusNone) return EBS_ERR_UNSUPPORTED;
    return check_cuda(cudaGraphLaunch(static_cast<cudaGraphExec_t>(graph_exec), st));
}

int ebs_graph_destroy(void* graph_exec) {
    if (!graph_exec) return EBS_ERR_INVALID_ARG;
    return check_cuda(cudaGraphExecDestroy(static_cast<cudaGraphExec_t>(graph_exec)));
}

}  // extern "C"
