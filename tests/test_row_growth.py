"""The row form of the 2D cluster moves (row_growth.cuh) in Python integers, lane
by lane, against a breadth-first search: count, reversal, seed in (colour,
site) order and component, for every shape, with rows that end inside a word,
lanes without rows, empty and full domains and wrapping runs."""
import random

import pytest

M=0xffffffff
K8,K16,K32,K64,K128=1,2,3,4,5
def shape(k): 
    FB={1:8,2:16}.get(k,32)
    U={1:2,2:8}.get(k,32)
    W={5:4,4:2}.get(k,1)
    return FB,U,W
def row_site(kind,j,i):
    fb={1:3,2:4}.get(kind,5)
    wl={5:2,4:1}.get(kind,0)
    return ((j&((1<<wl)-1))<<5)+(i&((1<<fb)-1)), ((j>>wl)<<(5-fb))+(i>>fb)
def popc(x): return bin(x).count('1')
def nth(v,r):
    for b in range(32):
        if (v>>b)&1:
            if r==0: return b
            r-=1
    assert 0
def fsr(lo,hi): return ((hi<<32|lo)>>1)&M
def sim(kind,L,neg,draw,en2a):
    FB,U,W=shape(kind)
    NW=W*W
    half=L*L//2
    nl=L//W if W>1 else -(-L//(32//FB))
    w=[[0]*NW for _ in range(U)]
    for j in range(U*NW):
        for i in range(32):
            x,y=row_site(kind,j,i)
            if x<L and y<L and neg[y][x]: w[j//NW][j%NW]|=1<<i
    def col0(ul,k):
        if FB==8: return 0xAA55AA55
        if FB==16: return 0xAAAA5555
        return 0xAAAAAAAA if ((ul if W==1 else k//W)&1) else 0x55555555
    n=sum(popc(x) for l in w for x in l)
    n0=sum(popc(w[u][k]&col0(u,k)) for u in range(U) for k in range(NW))
    flipped=en2a and 2*n>2*half
    if flipped:
        n=2*half-n
        n0=half-n0
        for u in range(U):
            for k in range(NW):
                if W>1:
                    left=L-32*(k%W) if u<nl else 0
                    valid=M if left>=32 else (1<<left)-1 if left>0 else 0
                else:
                    row=(M>>(32-FB)) if L==FB else (1<<L)-1
                    valid=0
                    for f in range(32//FB):
                        if u*(32//FB)+f<L: valid|=row<<(FB*f)
                w[u][k]=~w[u][k]&valid&M
    rank0=(draw*n)>>32
    second=rank0>=n0
    if second: rank0-=n0
    c=[[0]*NW for _ in range(U)]
    seed=-1
    incl=0
    for u in range(U):
        cnt=sum(popc(w[u][k]&((~col0(u,k) if second else col0(u,k))&M)) for k in range(NW))
        incl+=cnt
        rank=(rank0-(incl-cnt))&M
        at=-1
        for k in range(NW):
            v=w[u][k]&((~col0(u,k) if second else col0(u,k))&M)
            pc=popc(v)
            if at<0 and n>0 and rank<pc:
                at=k
                sel=v
                rr=rank
            if at<0: rank=(rank-pc)&M
        if incl<=0 or cnt==0: at=-1
        if at>=0:
            b=nth(sel,rr)
            c[u][at]=1<<b
            x,y=row_site(kind,u*NW+at,b)
            assert seed<0
            seed=y*L+x
    if W==1:
        RPW=32//FB
        lo={8:0x01010101,16:0x00010001,32:1}[FB]
        while True:
            old=[x[0] for x in c]
            new=[]
            for u in range(U):
                prv=nl-1 if u==0 else (u-1)&(U-1)
                nxt=0 if u>=nl-1 else u+1
                f=(L-1)%RPW if u==nl-1 else RPW-1
                fp=(L-1)%RPW if u==0 else RPW-1
                up=old[nxt]
                dn=old[prv]
                cc=old[u]
                m=w[u][0]
                v=(up|dn) if FB==32 else ((cc>>FB)|(up<<(FB*f))|(cc<<FB)|(dn>>(FB*fp)))&M
                cc|=m&v
                h=((cc<<1)&~lo)|((cc>>1)&~(lo<<(FB-1)))|((cc>>(L-1))&lo)|((cc&lo)<<(L-1))
                cc|=m&h&M
                if FB==32:
                    cc|=m&~(m+cc)&M
                    cc|=m&(cc>>1)
                new.append(cc)
            for u in range(U): c[u][0]=new[u]
            if new==old: break
    else:
        RPL=W
        bl=(L-1)&31
        last=(L-1)>>5
        def row(words, r):
            return words[r * W:(r + 1) * W]

        def run(u, r):
            cr, mr = row(c[u], r), row(w[u], r)
            t = sum(mr[j] << (32 * j) for j in range(W)) + sum(cr[j] << (32 * j) for j in range(W))
            c[u][r * W:(r + 1) * W] = [cr[j] | (mr[j] & ~(t >> (32 * j)) & M) for j in range(W)]

        def back(u, r):
            for _ in range(2):
                cr, mr = row(c[u], r), row(w[u], r)
                t = [fsr(cr[j], cr[j + 1] if j + 1 < W else 0) for j in range(W)]
                c[u][r * W:(r + 1) * W] = [cr[j] | (mr[j] & t[j]) for j in range(W)]

        def seam(u, r):
            cr, mr = row(c[u], r), row(w[u], r)
            wrap = ((cr[0] & 1) << bl) & M
            cr[0] |= mr[0] & ((cr[last] >> bl) & 1)
            cr[last] |= mr[last] & wrap
            c[u][r * W:(r + 1) * W] = cr

        while True:
            for it in range(3):
                nn = [row(c[nl - 1 if u == 0 else u - 1], RPL - 1) for u in range(U)]
                for u in range(U):
                    for r in range(RPL):
                        for j in range(W):
                            c[u][r * W + j] |= w[u][r * W + j] & (c[u][(r - 1) * W + j] if r else nn[u][j])
                        run(u, r)
                nn = [row(c[0 if u >= nl - 1 else u + 1], 0) for u in range(U)]
                for u in range(U):
                    for r in range(RPL - 1, -1, -1):
                        for j in range(W):
                            c[u][r * W + j] |= w[u][r * W + j] & (c[u][(r + 1) * W + j] if r < RPL - 1 else nn[u][j])
                        back(u, r)
            for u in range(U):
                for r in range(RPL):
                    seam(u, r)
            op=0
            for u in range(U):
                dn=c[(nl-1 if u==0 else u-1)][(RPL-1)*W:]
                up=c[(0 if u>=nl-1 else u+1)][:W]
                for r in range(RPL):
                    cr=c[u][r*W:(r+1)*W]
                    for j in range(W):
                        v=(c[u][(r-1)*W+j] if r else dn[j])|(c[u][(r+1)*W+j] if r<RPL-1 else up[j])
                        v|=((cr[j]<<1)&M)|((cr[j-1]>>31) if j else (cr[last]>>bl)&1)
                        v|=fsr(cr[j],cr[j+1] if j+1<W else 0)
                        if j==last: v|=((cr[0]&1)<<bl)&M
                        op|=v&w[u][r*W+j]&~cr[j]
            if not op: break
    out=set()
    for j in range(U*NW):
        for i in range(32):
            if (c[j//NW][j%NW]>>i)&1:
                x,y=row_site(kind,j,i)
                assert x<L and y<L
                out.add((x,y))
    return n,flipped,seed,out
def ref(L,neg,draw,en2a):
    s=[[neg[y][x] for x in range(L)] for y in range(L)]
    n=sum(map(sum,s))
    fl=en2a and 2*n>L*L
    if fl:
        s=[[1-v for v in r] for r in s]
        n=L*L-n
    if n==0: return 0,fl,-1,set()
    rank=(draw*n)>>32
    order=[(x,y) for col in (0,1) for y in range(L) for x in range(L) if (x+y)&1==col and s[y][x]]
    x,y=order[rank]
    seen={(x,y)}
    st=[(x,y)]
    while st:
        a,b=st.pop()
        for p in (((a+1)%L,b),((a-1)%L,b),(a,(b+1)%L),(a,(b-1)%L)):
            if s[p[1]][p[0]] and p not in seen:
                seen.add(p)
                st.append(p)
    return n,fl,y*L+x,seen


@pytest.mark.parametrize("kind,L,trials", [(K8, 2, 20), (K8, 4, 20), (K8, 6, 20), (K8, 8, 20), (K16, 10, 15), (K16, 14, 15),
                                           (K16, 16, 15), (K32, 18, 10), (K32, 30, 10), (K32, 32, 10), (K64, 34, 4),
                                           (K64, 62, 4), (K64, 64, 4), (K128, 68, 2), (K128, 100, 2), (K128, 128, 2)])
def test_rows_equal_breadth_first_search(kind, L, trials):
    rng = random.Random(L)
    for trial in range(trials):
        p = [0.5, 0.55, 0.0, 0.3, 0.62, 0.02, 0.9, 1.0][trial % 8]
        neg = [[1 if rng.random() < p else 0 for _ in range(L)] for _ in range(L)]
        draw, two_a = rng.choice([0, M, rng.getrandbits(32)]), rng.random() < 0.7
        a, b = sim(kind, L, neg, draw, two_a), ref(L, neg, draw, two_a)
        assert (a[0], bool(a[1]), a[2], a[3]) == (b[0], bool(b[1]), b[2], b[3])
