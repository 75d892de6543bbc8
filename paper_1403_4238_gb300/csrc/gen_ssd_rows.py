"""Writes ssd_rows.cuh: the inline-PTX row sequences of the engine's search.

One target row of the masked SSD (Sec. 3, Eq. 4) for the 4, 8 or 16 candidates
a lane owns: for each known target column c and candidate k, the byte-SIMD
absolute difference |t[c] - r[k + c]| (vabsdiff4) and its dot product with
itself accumulated into acc[k] (dp4a), i.e. the squared RGB distance of one
pixel pair.  A row whose known columns are [s, P) enters the ascending
sequence at column s; a row known on [0, e) enters the descending sequence at
column e - 1; both through one warp-uniform indexed branch (brx.idx) over a
table of 2P entries, so the row costs one jump instead of a test per column.
The caller passes an index in [0, 2P) (it clamps it).

The masked sequences (four candidates) also take a mask word per strip word,
ANDed to the difference: the partial-overlap search's rows with unavailable
source pixels.

The library build (paper_1403_4238_gb300/_lib.py) runs this script and
writes its output to the build directory, which is on the include path.
"""
NCLS = (4, 8, 16)  # candidates per lane (streaming: 4 or 8, resident: 4 or 16)
RADII = range(1, 9)


def row_macro(P: int, NCL: int, masked: bool = False) -> str:
    ns = (NCL + P - 1 + 3) & ~3   # strip words per lane
    tp = (P + 3) & ~3             # padded target row
    o_r, o_t = NCL, NCL + ns
    o_i = o_t + tp
    o_m = o_i + 1                 # masks, one per strip word
    lines = ["{", ".reg .b32 d, z;", "mov.b32 z, 0;"]
    labels = [f"Lra{c}" for c in range(P)] + [f"Lrd{c}" for c in range(P)]
    lines.append("Lrtab: .branchtargets " + ", ".join(labels) + ";")
    lines.append(f"brx.idx.uni %{o_i}, Lrtab;")

    def column(c):
        out = []
        for k in range(NCL):
            out.append(f"vabsdiff4.u32.u32.u32 d, %{o_t + c}, %{o_r + k + c}, z;")
            if masked:
                out.append(f"and.b32 d, d, %{o_m + k + c};")
            out.append(f"dp4a.u32.u32 %{k}, d, d, %{k};")
        return out

    for c in range(P):
        lines.append(f"Lra{c}:")
        lines += column(c)
    lines.append("bra.uni Lrend;")
    for c in range(P - 1, -1, -1):
        lines.append(f"Lrd{c}:")
        lines += column(c)
    lines.append("Lrend:")
    lines.append("}")
    body = "\\n\\t".join(lines)
    acc = ", ".join(f'"+r"(acc[{k}])' for k in range(NCL))
    ins = ", ".join([f'"r"(r[{i}])' for i in range(ns)] + [f'"r"(t[{i}])' for i in range(tp)] + ['"r"(idx)']
                    + ([f'"r"(m[{i}])' for i in range(ns)] if masked else []))
    name, args = (f"ROWM_P{P}", "acc, r, m, t, idx") if masked else (f"ROW{NCL}_P{P}", "acc, r, t, idx")
    return (f"// P = {P}: strip r[{ns}], target row t[{tp}], {NCL} accumulators\n"
            f"#define INP_SSD_{name}({args}) \\\n"
            f"  asm volatile(\"{body}\" \\\n"
            f"               : {acc} \\\n"
            f"               : {ins})\n")


def main():
    print("// Generated by gen_ssd_rows.py: inline-PTX row sequences of the engine's")
    print("// masked-SSD search, 4, 8 or 16 candidates per lane (see that script).  Do not edit.")
    print("#pragma once")
    print()
    for r in RADII:
        for ncl in NCLS:
            print(row_macro(2 * r + 1, ncl))
        print(row_macro(2 * r + 1, 4, masked=True))


if __name__ == "__main__":
    main()
