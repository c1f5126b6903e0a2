// The mesh deposit's volume of a polytope (mesh_volume), on polytopes written by hand: a cube
// with an edge of 2 about the origin, the same off the origin, and vertex lists that are no
// polytope (a vertex missing, a vertex twice). Prints one volume a line.
#include <cstdio>

#include "mesh.cu"

namespace sdot {
int num_sms() { return 1; }
void note_launch() {}
void set_error(const std::string&) {}
ClipParams mesh_clip_params(DeviceState&) { return ClipParams(); }
}  // namespace sdot

using namespace sdot;

constexpr int CASES = 4;

template <class C>
__global__ void volumes(double* out) {
    Poly<double, C>& P = poly_at<double, C>(0);
    const int lane = threadIdx.x;
    for (int k = 0; k < CASES; k++) {
        const double o[3] = {k == 1 ? 0.25 : 0.0, k == 1 ? -0.5 : 0.0, k == 1 ? 0.125 : 0.0};
        __syncwarp();
        if (lane < 6) {  // +x -x +y -y +z -z
            const int a = lane >> 1;
            const double s = (lane & 1) ? -1.0 : 1.0;
            P.pl[lane] = V4<double>{a == 0 ? s : 0.0, a == 1 ? s : 0.0, a == 2 ? s : 0.0,
                                    1.0 + s * o[a]};
            P.plen[lane] = 1.0;
            P.pj[lane] = mesh_tag(a, s > 0.0);
        }
        if (lane < 8) {  // corner (x, y, z), its planes ordered so that their normals turn right
            const int x = lane & 1, y = (lane >> 1) & 1, z = lane >> 2;
            const uint32_t a = x ? 0 : 1, b = y ? 2 : 3, c = z ? 4 : 5;
            P.tri[lane] = ((x + y + z) & 1) ? pack3(a, b, c) : pack3(a, c, b);
            P.vx[lane] = (x ? 1.0 : -1.0) + o[0];
            P.vy[lane] = (y ? 1.0 : -1.0) + o[1];
            P.vz[lane] = (z ? 1.0 : -1.0) + o[2];
        }
        if (lane == 0) {
            P.np = 6;
            P.nt = k == 2 ? 7 : 8;
        }
        __syncwarp();
        if (k == 3 && lane == 0) {  // vertex 7 again as vertex 8
            P.tri[8] = P.tri[7];
            P.vx[8] = P.vx[7];
            P.vy[8] = P.vy[7];
            P.vz[8] = P.vz[7];
            P.nt = 9;
        }
        __syncwarp();
        const double v = mesh_volume<C>(0, lane);
        if (lane == 0) out[k] = v;
    }
}

template <class C>
static int run(double* dev) {
    const int smem = (int)sizeof(Poly<double, C>);
    cudaFuncSetAttribute(volumes<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    volumes<C><<<1, 32, smem>>>(dev);
    double h[CASES];
    const cudaError_t e = cudaMemcpy(h, dev, sizeof h, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) {
        printf("error %s\n", cudaGetErrorString(e));
        return 1;
    }
    for (double v : h) printf("%.17g\n", v);
    return 0;
}

int main() {
    double* dev = nullptr;
    if (cudaMalloc(&dev, CASES * sizeof(double)) != cudaSuccess) return 1;
    const int rc = run<MeshCap>(dev) || run<CapL>(dev);
    cudaFree(dev);
    return rc;
}
