import sys
sys.path.insert(0,'/root/repo')
# max sum |c| into a destination, single and paired tables, by brute force on small widths
from collections import defaultdict
def canon(s):
    m={};return tuple(m.setdefault(x,len(m)) for x in s)
def oph(t,a,b):
    o=[]
    for s,c,sh in t:
        if s[a]==s[b]: continue
        o.append((s,c,sh)); o.append((canon([s[a] if x==s[b] else x for x in s]),-c,sh+1))
    return o
def opv(t,i):
    o=[]
    for s,c,sh in t:
        o.append((s,-c,sh+1)); l=list(s);l[i]=99;o.append((canon(l),c,sh))
    return o
def opd(t,i):
    o=[]
    for s,c,sh in t:
        l=list(s);l[i]=99;o.append((canon(l),c,sh))
    return o
def opp(t,lo,hi,skip): return [x for x in t if all(q==skip or x[0][q]!=x[0][q+1] for q in range(lo,hi))]
def fac(s,i,L,tri):
    t=[(s,1,0)]
    if not tri:
        if i<L-1:t=oph(t,i,i+1)
        t=opv(t,i);t=opp(t,0,L-1,i if i<L-1 else -1)
    else:
        if i<L-1:t=oph(t,i,i+1)
        if i>0:t=oph(t,i-1,i)
        t=opv(t,i);t=opp(t,0,L-1,-1)
    return t
def last(s,i,L):
    t=oph([(s,1,0)],i,i+1) if i<L-1 else [(s,1,0)]
    t=opd(t,i);return opp(t,i+1,L-1,-1)
for L in range(3,12):
  for tri in (0,1):
    st={tuple(range(L))}
    # closure over 3 rows approx
    spaces=[None]*(L+1)
    cur=st
    for row in range(6):
        for i in range(L):
            spaces[i]=(spaces[i] or set())|cur
            cur={x[0] for s in cur for x in fac(s,i,L,tri)}
    B=spaces[0]|cur
    res=[]
    for i in range(L):
        S=defaultdict(int);mx=0;E=defaultdict(int)
        for s in spaces[i]:
            for d,c,sh in fac(s,i,L,tri): S[d]+=abs(c);E[d]+=1
        P=defaultdict(int)
        if i+1<L:
            for s in spaces[i]:
                for d,c,sh in fac(s,i,L,tri):
                    for d2,c2,sh2 in fac(d,i+1,L,tri): P[d2]+=abs(c*c2)
        T=defaultdict(int)
        if i+2<L:
            for s in spaces[i]:
                for d,c,sh in fac(s,i,L,tri):
                    for d2,c2,sh2 in fac(d,i+1,L,tri):
                        for d3,c3,sh3 in fac(d2,i+2,L,tri): T[d3]+=abs(c*c2*c3)
        res.append((max(S.values()),max(P.values(),default=0),max(T.values(),default=0)))
    lr=[]
    cur=B
    for i in range(L-1):
        S=defaultdict(int);P=defaultdict(int)
        for s in cur:
            for d,c,sh in last(s,i,L):
                S[d]+=abs(c)
                if i+2<L:
                    for d2,c2,sh2 in last(d,i+1,L): P[d2]+=abs(c)
        lr.append((max(S.values()),max(P.values(),default=0)))
        cur=set(S)
    print(L,tri,len(B),"row",max(r[0] for r in res),max(r[1] for r in res),max(r[2] for r in res),"last",max(l[0] for l in lr),max(l[1] for l in lr))
