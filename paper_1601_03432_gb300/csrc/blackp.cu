#include "/root/repo/paper_1601_03432_gb300/csrc/smpm_device.cuh"
#include "/root/repo/paper_1601_03432_gb300/csrc/smpm_digits.cuh"
namespace {
#include "/root/repo/paper_1601_03432_gb300/csrc/smpm_gmres.cuh"
__global__ void __launch_bounds__(256,1) k(GmresArgs<double> a0, Smem<double> s0, BasisView<double> v0, double* o, int n){
  extern __shared__ unsigned char smraw[];
  __shared__ GmresArgs<double> a; __shared__ Smem<double> s; __shared__ BasisView<double> v;
  if(threadIdx.x==0){a=a0;s=s0;v=v0;}
  __syncthreads();
  unsigned ep=0; int tr=0;
  black_phase<double>(a,s,o,1.0,o);
}
}
const void* f(){return (const void*)k;}
