// gl_noalloc.cu -- gl_jacobian_apply_noalloc: the Jacobian apply of an existing
// mesh without any device allocation, for callers that cannot let a call allocate:
// applications that manage a fixed device-memory budget or their own pool (an
// allocation behind their back can fail or fragment it), and latency-critical
// loops (cudaMalloc/cudaFree can synchronise the device).
//
// It runs the kernel of gl_jacobian_apply in FP64, which works on the caller's
// node-order vectors and needs no buffer of its own.  Only where y lies partly over
// psi or phi is the result formed in a file-scope array first (4 MiB, shared by all
// such calls on a device: two of them must not overlap on the GPU).  Meshes beyond
// GL_NOALLOC_MAX_NODES are refused, as they always were.
#include "gl_internal.cuh"

// maximum number of mesh nodes this entry point accepts
#define GL_NOALLOC_MAX_NODES (1 << 18)

static __device__ double2 g_noalloc_y[GL_NOALLOC_MAX_NODES];

extern "C" gl_status gl_jacobian_apply_noalloc(gl_mesh m, const void *psi, const void *phi, void *y, void *stream) {
    try {
        gl::set_error("");
        GL_REQUIRE(m && psi && phi && y, GL_ERR_ARG, "NULL argument");
        GL_REQUIRE(y != psi && y != phi, GL_ERR_ARG, "y must not alias psi or phi");
        if (m->n > GL_NOALLOC_MAX_NODES)
            throw gl::Error{GL_ERR_CAPACITY, "gl_jacobian_apply_noalloc: mesh has " + std::to_string(m->n) +
                                                 " nodes, this entry point takes at most " +
                                                 std::to_string(GL_NOALLOC_MAX_NODES)};
        cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
        double2 *out = static_cast<double2 *>(y);
        const bool over = gl::overlap(y, psi, m->n) || gl::overlap(y, phi, m->n);
        if (over) GL_CUDA(cudaGetSymbolAddress(reinterpret_cast<void **>(&out), g_noalloc_y));
        gl::jacobian_apply_nodes(m, static_cast<const double2 *>(psi), static_cast<const double2 *>(phi), out, s);
        if (over) GL_CUDA(cudaMemcpyAsync(y, out, m->n * sizeof(double2), cudaMemcpyDeviceToDevice, s));
        return GL_OK;
    } catch (const gl::Error &e) {
        gl::set_error(e.msg);
        return e.code;
    } catch (const std::bad_alloc &) {
        gl::set_error("host allocation failed");
        return GL_ERR_OOM;
    } catch (const std::exception &e) {
        gl::set_error(e.what());
        return GL_ERR_CUDA;
    }
}
