// Rows of the exchange buffer ([kCgRows][CTAs], one partial sum per CTA) that the
// reductions of the one-kernel Schur CG (resident.cu) use.  A reduction is: every CTA
// writes its entry of the rows, all meet, every CTA reads the rows.  A CTA may leave
// that meeting and write the rows of the next reduction while another still reads, so
// two reductions with no other meeting between them need rows of their own: p . q and
// the r . r, r . z that follow it.  The operator, with one to three meetings, lies
// between the others (start and p . q, r . z and the next p . q).
#pragma once

struct CgSums {
    int row, n;
};
constexpr int kCgRows = 3;
constexpr CgSums kCgStart{0, 3};   // r . z, g . g, r . r before the first iteration
constexpr CgSums kCgRes{0, 2};     // r . r, r . z of an iteration
constexpr CgSums kCgPq{2, 1};      // p . q
static_assert(kCgPq.row >= kCgRes.row + kCgRes.n || kCgRes.row >= kCgPq.row + kCgPq.n, "no meeting between these two");
static_assert(kCgStart.row + kCgStart.n <= kCgRows && kCgRes.row + kCgRes.n <= kCgRows && kCgPq.row + kCgPq.n <= kCgRows,
              "rows of the buffer");
