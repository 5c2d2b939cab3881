// Host driver for the double-float arithmetic of csrc/df.cuh (compiled by
// tests/test_df_host.py with the host compiler): reads lines of an operation
// and hexadecimal numbers and prints the result's as hexadecimal numbers, so
// that the test can check each step against exact rational arithmetic.
//   split d         -> the pair of df_split, then that of DF(d)
//   widen f         -> df_widen
//   add|sub|mul2|cmul|cscale|cfma  a b c -> result
// where each complex operand is re.hi re.lo im.hi im.lo, and so is the result
// (cscale multiplies a by the real part of b).
#include <cstdio>
#include <cstring>

#include "df.cuh"

using namespace dda;

static cdf read_cdf() {
    double v[4];
    for (double& x : v)
        if (std::scanf("%la", &x) != 1) x = 0.0;
    return make_cdf(DF((float)v[0], (float)v[1]), DF((float)v[2], (float)v[3]));
}

int main() {
    char op[16];
    while (std::scanf("%15s", op) == 1) {
        double d;
        if (!std::strcmp(op, "split")) {
            if (std::scanf("%la", &d) != 1) return 2;
            const DF a = df_split(d), b(d);
            std::printf("%a %a %a %a\n", (double)a.hi, (double)a.lo, (double)b.hi, (double)b.lo);
            continue;
        }
        if (!std::strcmp(op, "widen")) {
            if (std::scanf("%la", &d) != 1) return 2;
            std::printf("%a\n", df_widen((float)d));
            continue;
        }
        const cdf a = read_cdf(), b = read_cdf(), c = read_cdf();
        cdf r;
        if (!std::strcmp(op, "add")) r = df_add(a, b);
        else if (!std::strcmp(op, "sub")) r = df_sub(a, b);
        else if (!std::strcmp(op, "mul2")) r = df_mul2(a.h, a.l, b.h, b.l);
        else if (!std::strcmp(op, "cmul")) r = df_cmul(a, b);
        else if (!std::strcmp(op, "cscale")) r = df_cscale(a, DF(b.h.x, b.l.x));
        else if (!std::strcmp(op, "cfma")) r = df_cfma(a, b, c);
        else return 2;
        std::printf("%a %a %a %a\n", (double)r.h.x, (double)r.l.x, (double)r.h.y, (double)r.l.y);
    }
    return 0;
}
