#include <cstdio>
#include "fft_mixed.cuh"
using namespace bplg::mixed_detail;
void pr(const char*t,int n,const Plan&p){ printf("%s n=%d k=%d r=",t,n,p.k); for(int i=0;i<p.k;++i)printf("%d ",p.r[i]); printf("pitch="); for(int i=0;i+1<p.k;++i)printf("%d ",p.pitch[i]); printf("t=%d b=%d spb=%d threads=%d minb=%d vmax=%d dbl=%d sig=%d sig2=%d smem/SM=%d\n",p.t,p.b,p.spb,p.threads,p.minb,p.vmax,p.dbl,p.sig,p.sig2,smem_per_sm(p)); }
int cost(int m,int mn,int pitch,int*a,int*b){int c=0;*a=*b=0; for(int t0=0;t0<240;t0+=16){*a+=half_warp_wavefronts(t0,m,pitch);*b+=half_warp_wavefronts(t0,mn,pitch);} return *a+*b;}
int main(){ for(int n:{216,108,360,180,432,1080}){ pr("pad ",n,plan_of(n,kNumWide,true)); pr("nop ",n,plan_of(n,kNumWide,false)); pr("kern",n,kernel_plan(n)); }
 for(int p=36;p<52;++p){int a,b;int c=cost(36,6,p,&a,&b);printf("pitch %d: %d (w %d r %d)\n",p,c,a,b);} for(int p=6;p<=7;++p){int a,b;int c=cost(6,1,p,&a,&b);printf("m6 pitch %d: %d (w %d r %d)\n",p,c,a,b);} 
 int cnt=0; for(int i=0;i<kNumLengths;++i){int n=kLengths.v[i];Plan p=kernel_plan(n); for(int s=0;s+1<p.k;++s){int rows=1; for(int q=0;q<=s;++q)rows*=p.r[q]; if(p.pitch[s]!=n/rows){cnt++; printf("%d:s%d %d->%d  ",n,s,n/rows,p.pitch[s]);}}} printf("\n%d\n",cnt);}
