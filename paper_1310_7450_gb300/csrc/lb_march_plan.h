// lb_march_plan.h -- the row-march kernel's work items (host arithmetic only: no CUDA header, so it also
// compiles and is tested without nvcc).
#pragma once

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <vector>

namespace lbk {

constexpr int kMarchW = 128;  // columns per CTA (one strip)

struct MarchItem {
    int x0, y0, y1;  // first column, rows [y0, y1)
    int w;           // columns (kMarchW at most)
};

// Width of a channel's strips: a multiple of 8 columns, the same for all but the last, which has two at least (a halo
// column's populations come from one column further on).  0: none does (nx - 1 a multiple of 5765760, which
// all of 8, 16, ... 128 divide).
inline int march_strip_width(int nx) {
    const int least = (nx + kMarchW - 1) / kMarchW;
    int W = std::min(kMarchW, ((nx + least - 1) / least + 7) / 8 * 8);
    while (W > 0 && nx % W == 1) W -= 8;
    return W;
}

// Row-march work items: strips of kMarchW columns cut into row ranges, at most one item per
// resident CTA (one wave: a partial second wave would double the kernel time for a few CTAs).
// Items are not equally long, because CTAs are not equally fast: the warp schedulers favour older
// warps, so the CTAs that arrive later on an SM take longer for the same rows, and an edge strip costs more per row than an interior one (its
// halo columns are patched from the other end; with pressure-driven ends it also applies the
// crossing corrections).  The model: block b, of rank k = b / n_sm (blocks fill the SMs rank by
// rank), runs at speed 1 + skew (R-1-k)/(R-1) for R CTAs per SM; strip j costs f_j per row (f for
// the two edge strips, 1 inside).  A bisection finds the smallest common duration T whose dealing
// needs at most R n_sm blocks; rows are then split in proportion to the blocks' speeds.  Two
// dealings:
//  - strip-major: each strip takes consecutive blocks until their speeds cover ny f_j / T;
//  - chunk-major: the edge strips first, the same way, then the interior strips share their row
//    boundaries -- row chunk c of every interior strip on consecutive blocks, T times the speed of
//    the slowest of them in rows -- so neighbouring strips march the same rows at the same time
//    and read each other's halo columns from L2 (with boundaries that differ between strips, BF16
//    re-reads 9 DRAM bytes per node of halo).  Both precisions are dealt chunk-major; strip-major
//    serves grids of one or two strips.
// Items keep at least 8 rows on average (at most ny / 8 per strip).
struct MarchModel {
    double skew, fedge;
    bool chunk_major;
};

inline std::vector<MarchItem> march_plan(int nx, int ny, int R, int nsm, MarchModel m) {
    const int W = march_strip_width(nx);
    const int strips = (nx + W - 1) / W;
    auto width = [&](int x0) { return std::min(W, nx - x0); };
    const int slots = R * nsm;
    const int maxn = std::max(1, ny / 8);
    auto speed = [&](int b) {
        const int k = std::min(b / nsm, R - 1);
        return 1.0 + (R > 1 ? m.skew * (R - 1 - k) / (R - 1) : 0.0);
    };
    auto cost = [&](int s) { return (s == 0 || s == strips - 1) ? m.fedge : 1.0; };
    // the rows [0, ny) of one strip split in proportion to the weights w
    auto split = [&](std::vector<MarchItem>& out, int x0, const std::vector<double>& w) {
        double tot = 0.0;
        for (double v : w) tot += v;
        double cum = 0.0;
        int y = 0;
        for (size_t k = 0; k < w.size(); ++k) {
            cum += w[k];
            const int y1 = k + 1 == w.size() ? ny : (int)std::llround(ny * cum / tot);
            MarchItem it{};
            it.x0 = x0;
            it.y0 = y;
            it.y1 = y1;
            it.w = width(x0);
            out.push_back(it);
            y = y1;
        }
    };
    // blocks from b on until their speeds cover ny f / T (at most maxn)
    auto take = [&](double T, int b, double f) {
        double acc = 0.0;
        int n = 0;
        while (n < maxn && acc < ny * f / T) acc += speed(b + n++);
        return n;
    };
    const bool cm = m.chunk_major && strips >= 3 && strips < slots;
    const int I = strips - 2;
    // blocks per strip (strip-major) or [edge 0, edge 1, chunks] (chunk-major) at duration T
    auto deal = [&](double T, std::vector<int>* out) {
        int b = 0;
        if (!cm) {
            for (int s = 0; s < strips; ++s) {
                const int n = strips >= slots ? 1 : take(T, b, cost(s));
                if (out) out->push_back(n);
                b += n;
            }
            return b;
        }
        for (int e = 0; e < 2; ++e) {
            const int n = take(T, b, m.fedge);
            if (out) out->push_back(n);
            b += n;
        }
        int C = 0;
        double acc = 0.0;
        while (C < maxn && acc < ny) acc += T * speed(b + (++C) * I - 1);
        if (out) out->push_back(C);
        return b + C * I;
    };
    double lo = 1e-9, hi = 4.0 * ny * std::max(1.0, m.fedge);  // deal(hi): one block per strip
    if (strips >= slots || deal(lo, nullptr) <= slots) {
        hi = strips >= slots ? hi : lo;
    } else {
        for (int it = 0; it < 100; ++it) {
            const double mid = 0.5 * (lo + hi);
            if (deal(mid, nullptr) <= slots) hi = mid;
            else lo = mid;
        }
    }
    std::vector<int> n;
    deal(hi, &n);
    std::vector<MarchItem> items;
    int b = 0;
    auto strip_items = [&](int s, int cnt) {
        std::vector<double> w(cnt);
        for (int k = 0; k < cnt; ++k) w[k] = speed(b + k);
        split(items, s * W, w);
        b += cnt;
    };
    if (!cm) {
        for (int s = 0; s < strips; ++s) strip_items(s, n[s]);
        return items;
    }
    strip_items(0, n[0]);
    strip_items(strips - 1, n[1]);
    const int C = n[2];
    std::vector<double> wc(C);
    for (int c = 0; c < C; ++c) wc[c] = speed(b + (c + 1) * I - 1);
    std::vector<MarchItem> chunk;
    split(chunk, 0, wc);
    for (int c = 0; c < C; ++c)
        for (int s = 1; s <= I; ++s) {
            MarchItem it = chunk[c];
            it.x0 = s * W;
            it.w = width(it.x0);
            items.push_back(it);
        }
    return items;
}

// A grid too small to give every resident CTA an 8-row item is cut finer, down to 2 rows: a row takes about 1.5 us
// whatever the chip's load (its instructions wait for one another), so the launch lasts as long as its
// longest item.  128 x 512 FP32: 18.8 us with 8-row items, 9.6 with 2-row ones.
inline std::vector<MarchItem> fine_items(std::vector<MarchItem> in, int nx, int ny, int slots) {
    int strips = 0, W = in[0].w;
    for (const MarchItem& it : in) {
        strips += it.y0 == 0;
        W = std::max(W, it.w);
    }
    if ((long long)strips * (ny / 8) >= slots) return in;
    const int n = std::min(ny / 2, std::max(1, slots / strips));
    std::vector<MarchItem> out;
    for (int k = 0; k < n; ++k)
        for (int s = 0; s < strips; ++s) {
            MarchItem it{};
            it.x0 = s * W;
            it.w = std::min(W, nx - it.x0);
            it.y0 = (int)((long long)ny * k / n);
            it.y1 = (int)((long long)ny * (k + 1) / n);
            out.push_back(it);
        }
    return out;
}

// The kernel addresses an item's rows with 32-bit offsets: items of 2^29 elements or more are halved.
inline std::vector<MarchItem> short_items(const std::vector<MarchItem>& in, int nx) {
    std::vector<MarchItem> out;
    for (MarchItem it : in) {
        const long long most = std::max(8LL, (1LL << 29) / nx);
        while (it.y1 - it.y0 > most) {
            MarchItem a = it;
            a.y1 = it.y0 + (it.y1 - it.y0) / 2;
            it.y0 = a.y1;
            while (a.y1 - a.y0 > most) {
                MarchItem b = a;
                b.y1 = a.y0 + (int)most;
                out.push_back(b);
                a.y0 = b.y1;
            }
            out.push_back(a);
        }
        out.push_back(it);
    }
    return out;
}

}  // namespace lbk
