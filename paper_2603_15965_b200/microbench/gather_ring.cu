// Micro-benchmark (stand-alone, not part of the library): what the memory delivers for the tcgen05 apply's access pattern -- tiles of 128
// gathered rows, x read and then y read and written in pieces of 128 or 256 bytes per row through a ring of cp.async stages, stores of 32
// bytes per lane -- without arithmetic.  "hint": the copies carry .L2::256B.  Every wait is bounded.
//   nvcc -gencode arch=compute_100a,code=sm_100a -O3 -o gather_ring gather_ring.cu && ./gather_ring
#include <cuda_runtime.h>
#include <stdio.h>
#include <stdint.h>
#include <vector>
#include <random>
#include <algorithm>
#define CK(x) do{cudaError_t e=(x); if(e!=cudaSuccess){printf("err %s line %d\n",cudaGetErrorString(e),__LINE__);return 1;}}while(0)
__device__ __forceinline__ uint32_t s32(const void*p){return (uint32_t)__cvta_generic_to_shared(p);}
__device__ __forceinline__ void mbi(uint32_t b,uint32_t c){asm volatile("mbarrier.init.shared.b64 [%0], %1;"::"r"(b),"r"(c):"memory");}
__device__ __forceinline__ void mba(uint32_t b){asm volatile("mbarrier.arrive.shared.b64 _, [%0];"::"r"(b):"memory");}
__device__ __forceinline__ bool mbt(uint32_t b,uint32_t p){uint32_t ok;asm volatile("{.reg .pred p; mbarrier.try_wait.parity.shared.b64 p, [%1], %2; selp.u32 %0,1,0,p;}":"=r"(ok):"r"(b),"r"(p):"memory");return ok;}
__device__ bool wt(uint32_t b,uint32_t p,int*fail){ if(mbt(b,p))return true; long long t0=clock64(); while(!mbt(b,p)){ if(clock64()-t0>400000000LL){*fail=1;return false;} } return true;}
template<int PIECE,int HINT> __global__ void __launch_bounds__(256,1) k(const char* x, char* y, const int* perm, int tiles, int rowb, int ns, int* fail)
{
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ uint64_t full[16],empty[16];
  constexpr int ST=128*PIECE, LPR=PIECE/16; // lanes per row
  int tid=threadIdx.x, n=rowb/PIECE;
  if(tid==0){for(int i=0;i<ns;i++){mbi(s32(&full[i]),128);mbi(s32(&empty[i]),4);}asm volatile("fence.mbarrier_init.release.cluster;":::"memory");}
  __syncthreads();
  if(tid<128){
    constexpr int RPT=128*LPR/128; // rows per thread = LPR... 16B pieces per thread
    int s=0; uint32_t ph=1;
    for(int t=blockIdx.x;t<tiles;t+=gridDim.x){
      size_t off[RPT];
      #pragma unroll
      for(int i=0;i<RPT;i++) off[i]=(size_t)perm[t*128+tid/LPR+i*(128/LPR)]*rowb+(tid%LPR)*16;
      for(int c=0;c<2*n;c++){
        if(!wt(s32(&empty[s]),ph,fail)) return;
        const char* src=c<n? x+(size_t)c*PIECE : y+(size_t)(c-n)*PIECE;
        #pragma unroll
        for(int i=0;i<RPT;i++){ uint32_t d=s32(sm)+s*ST+(tid/LPR+i*(128/LPR))*PIECE+(((tid%LPR)^(((tid/LPR))&7))*16);
          if(HINT) asm volatile("cp.async.cg.shared.global.L2::256B [%0],[%1],16;"::"r"(d),"l"(src+off[i]):"memory"); else
          asm volatile("cp.async.cg.shared.global [%0],[%1],16;"::"r"(d),"l"(src+off[i]):"memory"); }
        asm volatile("cp.async.mbarrier.arrive.noinc.shared.b64 [%0];"::"r"(s32(&full[s])):"memory");
        if(++s==ns){s=0;ph^=1;}
      }
    }
  } else {
    int w=(tid-128)/32, lane=tid&31; int s=0; uint32_t ph=0;
    constexpr int L32=PIECE/32; // lanes per row with 32B
    constexpr int IT=32*L32/32;
    for(int t=blockIdx.x;t<tiles;t+=gridDim.x){
      size_t off[IT];
      #pragma unroll
      for(int i=0;i<IT;i++) off[i]=(size_t)perm[t*128+w*32+lane/L32+i*(32/L32)]*rowb+(lane%L32)*32;
      for(int c=0;c<2*n;c++){
        if(!wt(s32(&full[s]),ph,fail)) return;
        if(c>=n){
          uint4 a[IT],b[IT];
          #pragma unroll
          for(int i=0;i<IT;i++){ int r=w*32+lane/L32+i*(32/L32); int p0=(lane%L32)*2; const unsigned char* q=sm+s*ST+r*PIECE; a[i]=*(const uint4*)(q+((p0^(r&7))%LPR)*16); b[i]=*(const uint4*)(q+(((p0+1)^(r&7))%LPR)*16); }
          #pragma unroll
          for(int i=0;i<IT;i++) asm volatile("st.global.v8.b32 [%0],{%1,%2,%3,%4,%5,%6,%7,%8};"::"l"(y+off[i]+(size_t)(c-n)*PIECE),"r"(a[i].x),"r"(a[i].y),"r"(a[i].z),"r"(a[i].w),"r"(b[i].x),"r"(b[i].y),"r"(b[i].z),"r"(b[i].w):"memory");
        }
        __syncwarp();
        if(lane==0) mba(s32(&empty[s]));
        if(++s==ns){s=0;ph^=1;}
      }
    }
  }
}
template<int P,int H> int run(const char*name,char*x,char*y,int*dp,int N,int rowb,int ns,int*f){
  CK(cudaFuncSetAttribute(k<P,H>,cudaFuncAttributeMaxDynamicSharedMemorySize,200*1024));
  cudaEvent_t e0,e1; cudaEventCreate(&e0);cudaEventCreate(&e1); float best=1e9;
  for(int r=0;r<5;r++){CK(cudaEventRecord(e0)); k<P,H><<<148,256,ns*128*P>>>(x,y,dp,N/128,rowb,ns,f); CK(cudaEventRecord(e1)); CK(cudaEventSynchronize(e1)); float ms; cudaEventElapsedTime(&ms,e0,e1); best=std::min(best,ms);} 
  printf("%s row %d piece %d hint %d stages %d (%d KB): %.0f GB/s\n",name,rowb,P,H,ns,ns*128*P/1024,3.0*N*rowb/best/1e6); return 0; }
int main(){
  for(int rowb: {8192,4096}){
  int N=148*128*4; char*x,*y; CK(cudaMalloc(&x,(size_t)N*rowb)); CK(cudaMalloc(&y,(size_t)N*rowb)); CK(cudaMemset(x,0,(size_t)N*rowb)); CK(cudaMemset(y,0,(size_t)N*rowb));
  int*f; CK(cudaMalloc(&f,4)); CK(cudaMemset(f,0,4)); int*dp; CK(cudaMalloc(&dp,N*4));
  for(int rnd=0;rnd<2;rnd++){
    std::vector<int> p(N); for(int i=0;i<N;i++)p[i]=i; std::mt19937 g(1);
    if(rnd==1){ std::vector<int> q; std::vector<int> a(N); for(auto&v:a)v=g()%16; for(int c=0;c<16;c++)for(int i=0;i<N;i++)if(a[i]==c)q.push_back(i); p=q; }
    CK(cudaMemcpy(dp,p.data(),N*4,cudaMemcpyHostToDevice));
    const char*nm=rnd?"seg16":"seq";
    for(int ns: {4,7,9,12}){ run<128,0>(nm,x,y,dp,N,rowb,ns,f); run<128,1>(nm,x,y,dp,N,rowb,ns,f); }
    for(int ns: {3,4,6}){ run<256,0>(nm,x,y,dp,N,rowb,ns,f); run<256,1>(nm,x,y,dp,N,rowb,ns,f);}
  }
  int h; CK(cudaMemcpy(&h,f,4,cudaMemcpyDeviceToHost)); printf("fail %d\n",h); cudaFree(x);cudaFree(y);cudaFree(dp);}
}
