"""Generate m2l_unrolled.cuh: straight-line MtL contraction bodies for fixed Taylor orders.

For a fixed order P the MtL sum of eqcoeff, written as
    a! lam^a = sum_{|a| + |b| <= P} D^{a+b} G(d) * M^b,   M^b = (-1)^|b| m^b / b!,
has a fixed set of (gamma = a + b, a, b) triples. Emitting them as explicit statements lets
the compiler keep the local coefficients in registers. M2LBody<P, W> (FP64 kernel) handles one of
NBODY[P] sets of multi-indices a with equal FMA counts (at most 43 coefficients, so that a set's
accumulators fit in registers), walks gamma in layout order, loads D^gamma from the interleaved
slot layout (Dl[gamma * 32]) in groups of GROUP so that several loads are in flight before their
values are used, and reads the scaled moments from shared memory (Ms[b * 33]) for every FMA
(volatile: kept in registers across FMAs they spilled the accumulators).

M2LWarp<P, W> is the register-blocked two-warp variant used by the FP32 kernel: warp W
accumulates half of the local coefficients (equal FMA counts) and the moments of a block of
MBLOCK multi-indices sit in registers. Derivatives and moments come four at a time (16-byte
shared-memory loads): four consecutive gammas of a slot lie together (Dl[gamma / 4 * 32], a float4
per lane), and a lane's moments are a row of its own (Ms[b / 4]). 168 loads for 3003 FMAs at P = 8,
both warps together, about 170 registers per thread and no spills.

Run: python gen_m2l.py > m2l_unrolled.cuh  (the output is committed beside this script).
"""

from math import comb

ORDERS = (4, 6, 8)
NBODY = {4: 1, 6: 2, 8: 4}
GROUP = 4
# two-warp register-blocked bodies (FP32 kernel): the local coefficients are split between two
# warps with equal FMA counts, and each warp holds the moments of MBLOCK multi-indices at a
# time in registers
NWARP = 2
MBLOCK = {4: 36, 6: 84, 8: 84}  # multiples of 4
# row stride of the moments in shared memory of the FP64 kernel: 33, so that it can write one
# source's moments (lanes over b) without bank conflicts
MSTRIDE = 33


def multi_indices(p):
    out = []
    for n in range(p + 1):
        for a in range(n, -1, -1):
            for b in range(n - a, -1, -1):
                out.append((a, b, n - a - b))
    return out


def body(P, aset):
    idx = multi_indices(P)
    pos = {t: i for i, t in enumerate(idx)}
    work = []  # (gamma, [(k, beta)])
    for g, gm in enumerate(idx):
        splits = []
        for k, ia in enumerate(aset):
            al = idx[ia]
            be = (gm[0] - al[0], gm[1] - al[1], gm[2] - al[2])
            if min(be) >= 0:
                splits.append((k, pos[be]))
        if splits:
            work.append((g, splits))
    out = []
    for s in range(0, len(work), GROUP):
        grp = work[s:s + GROUP]
        for k, (g, _) in enumerate(grp):
            out.append(f"        d{k} = Dl[{g * 32}];")
        for k, (_, splits) in enumerate(grp):
            for ia, ib in splits:
                out.append(f"        L[{ia}] += d{k} * Ms[{ib * MSTRIDE}];")
    return out


def warp_sets(P, nwarp=NWARP):
    """Split the multi-indices a between nwarp warps so that each gets the same number of
    (a, b) pairs: a pairs with C(P - |a| + 3, 3) moments, so low orders are heavy. Greedy,
    heaviest first, ties to the lower warp; each set in layout order."""
    idx = multi_indices(P)
    wt = [comb(P - sum(a) + 3, 3) for a in idx]
    load = [0] * nwarp
    sets = [[] for _ in range(nwarp)]
    for i in sorted(range(len(idx)), key=lambda i: (-wt[i], i)):
        k = load.index(min(load))
        load[k] += wt[i]
        sets[k].append(i)
    return [sorted(x) for x in sets]


def quad(src, names):
    """One 16-byte load into the named variables (None: not needed)."""
    out = [f"        v = {src};"]
    return out + [f"        {n} = v.{c};" for n, c in zip(names, "xyzw") if n]


def body_blocked(P, mb, aset):
    """Register-blocked form for the local coefficients a in `aset` (held as L[k], k the
    position in aset): the moments M^b of one block of mb multi-indices are loaded into
    registers once; then each D^gamma that pairs with the block is loaded once and every
    pair (a = gamma - b in aset, b in the block) is accumulated. Shared-memory loads per slot
    drop from one per FMA to (#gamma reached per block) + (#moments used)."""
    idx = multi_indices(P)
    pos = {t: i for i, t in enumerate(idx)}
    loc = {a: k for k, a in enumerate(aset)}
    T = len(idx)
    out = []
    for b0 in range(0, T, mb):
        blk = list(range(b0, min(T, b0 + mb)))
        work, used = [], set()
        for g, gm in enumerate(idx):
            prs = []
            for k, b in enumerate(blk):
                be = idx[b]
                al = (gm[0] - be[0], gm[1] - be[1], gm[2] - be[2])
                if min(al) >= 0 and pos[al] in loc:
                    prs.append((loc[pos[al]], k))
                    used.add(k)
            if prs:
                work.append((g, prs))
        for k in sorted({k // 4 for k in used}):  # (blk[0] is a multiple of 4)
            names = [f"m{4 * k + j}" if 4 * k + j in used else None for j in range(4)]
            out += quad(f"Ms[{blk[0] // 4 + k}]", names)
        for g4 in sorted({g // 4 for g, _ in work}):
            grp = [(g, prs) for g, prs in work if g // 4 == g4]
            live = {g % 4 for g, _ in grp}
            out += quad(f"Dl[{g4 * 32}]", [f"d{j}" if j in live else None for j in range(4)])
            for g, prs in grp:
                for ia, km in prs:
                    out.append(f"        L[{ia}] += d{g % 4} * m{km};")
    return out


def main():
    lines = [
        "// Generated by gen_m2l.py -- straight-line MtL contraction bodies. Do not edit.",
        "#pragma once",
        "",
        "// FP64 bodies: the sets of local coefficients (warps) and the largest set",
        "template <int P>",
        "struct M2LBodies;",
        "template <int P, int W>",
        "struct M2LBody;",
        "",
    ]
    for P in ORDERS:
        sets = warp_sets(P, NBODY[P])
        lines.append(f"template <>\nstruct M2LBodies<{P}> {{\n    static constexpr int n = {NBODY[P]}, "
                     f"most = {max(map(len, sets))};\n}};\n")
        for w, aset in enumerate(sets):
            lines += [
                "template <>",
                f"struct M2LBody<{P}, {w}> {{",
                f"    static constexpr int n = {len(aset)};",
                "    static __device__ __forceinline__ int alpha(int k)",
                "    {",
                f"        constexpr short a[{len(aset)}] = {{{', '.join(str(x) for x in aset)}}};",
                "        return a[k];",
                "    }",
                "    template <class R>",
                "    static __device__ __forceinline__ void run(const R* __restrict__ Dl, const volatile R* Ms, R* L)",
                "    {",
                "        R " + ", ".join(f"d{i}" for i in range(GROUP)) + ";",
            ]
            lines += body(P, aset)
            lines += ["    }", "};", ""]
    lines += ["template <int P, int W>", "struct M2LWarp;", ""]
    for P in ORDERS:
        mb = MBLOCK[P]
        for w, aset in enumerate(warp_sets(P)):
            text = body_blocked(P, mb, aset)
            ms = {ln.split()[0] for ln in text if ln.split()[0][0] == "m"}
            lines += [
                "template <>",
                f"struct M2LWarp<{P}, {w}> {{",
                f"    static constexpr int n = {len(aset)};",
                "    // the local-coefficient multi-indices this warp accumulates, in order",
                "    static __device__ __forceinline__ int alpha(int k)",
                "    {",
                f"        constexpr short a[{len(aset)}] = {{{', '.join(str(x) for x in aset)}}};",
                "        return a[k];",
                "    }",
                "    static __device__ __forceinline__ void run(const float4* __restrict__ Dl, const float4* __restrict__ Ms,",
                "                                               float* L)",
                "    {",
                "        float4 v;",
                "        float " + ", ".join(sorted(ms, key=lambda m: int(m[1:]))) + ";",
                "        float " + ", ".join(f"d{i}" for i in range(GROUP)) + ";",
            ]
            lines += text
            lines += ["    }", "};", ""]
    print("\n".join(lines))


if __name__ == "__main__":
    main()
